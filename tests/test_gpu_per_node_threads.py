"""Per-node contractions of two handles from two host threads. The kernel's dynamic shared memory follows the
handle's quadrature points M and n_pl (98 KB at M = 6144, 1 KB at M = 64), and its limit belongs to the
function, not the launch: a handle that lowered it between another's setting and launch made that launch fail.
Each thread's results equal its first ones (the kernel has no atomics): no tolerance."""
import threading

import numpy as np
import pytest

from workloads import tiny_instance

pytestmark = pytest.mark.gpu


def test_contractions_of_different_sizes_run_side_by_side():
    import torch
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq
    insts = [dict(tiny_instance(seed=3, n=(4, 4, 3), h=(0.7, 0.7, 0.7), n_atoms=1, n_o=2, r_cut=1.5, n_pl=6), M=m)
             for m in (6144, 64)]
    streams = [torch.cuda.Stream() for _ in insts]
    hs = [sq.sq_setup(sq.Desc(i, sq.SQ_FP64, bounds="per_node", stream=s.cuda_stream)) for i, s in zip(insts, streams)]
    errors = []
    try:
        first = []
        for h in hs:
            sq.sq_moments(h)
            mu = sq.sq_fermi_level(h)
            first.append((mu, sq.sq_density_energy_stress(h, mu)))
        start = threading.Barrier(len(hs))

        def work(h, mu, ref):
            try:
                start.wait()
                for _ in range(4000):
                    _, en, sig = sq.sq_density_energy_stress(h, mu)
                    assert en == ref[1] and np.array_equal(sig, ref[2])
            except Exception as e:   # reported by the main thread
                errors.append(e)

        pool = [threading.Thread(target=work, args=(h, mu, ref)) for h, (mu, ref) in zip(hs, first)]
        for t in pool:
            t.start()
        for t in pool:
            t.join()
        assert not errors, errors
    finally:
        for h in hs:
            sq.sq_destroy(h)
