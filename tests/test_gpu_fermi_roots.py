"""The Fermi level where N(mu) = N_e has several roots: the truncated expansion of a few narrow levels with cold
smearing makes N(mu) rise and fall, and the level is the root that bisection from the whole bracket ends in
(the oracle's rule), not another one.

Tolerance as in test_gpu_fermi.py: the last interval is 1e-13 max(1, |mu|) wide, and N' >= 1.4 at these roots with
N's rounding at 1e-14 or so: 1e-11 covers both."""
import numpy as np
import pytest

from oracle import sq_oracle as orc
from workloads import tiny_instance

pytestmark = pytest.mark.gpu

ND, N_PL, KT = 48, 56, 0.02


def _node_sums(seed):
    x = np.random.default_rng(seed).uniform(-0.9, 0.9, 4)
    return ND * np.cos(np.outer(np.arange(N_PL + 1), np.arccos(x))).mean(axis=1)


@pytest.mark.parametrize("seed,filling", [(0, 0.49), (1, 0.25), (1, 0.49), (2, 0.25), (4, 0.25), (8, 0.77), (11, 0.49),
                                          (14, 0.49), (16, 0.25)])
def test_the_bisections_root_of_several(seed, filling):
    from paper_2006_03697_gb300 import build
    build.build()
    import torch
    from paper_2006_03697_gb300 import sq
    inst = tiny_instance(seed=21, n=(4, 4, 3), h=(0.7, 0.7, 0.7), n_atoms=1, n_o=1, r_cut=0.8, n_pl=N_PL, kT=KT, M=2048)
    inst["n_e"] = 2 * ND * filling
    R = _node_sums(seed)
    h = sq.sq_setup(sq.Desc(inst, sq.SQ_FP64, bounds=(-6.0, 12.0)))
    try:
        lo, hi = sq.sq_get_bounds(h)
        mu = sq.sq_fermi_level_sums(h, R)
    finally:
        sq.sq_destroy(h)
    ref = orc.fermi_bisect(R, inst["n_e"], KT, lo, hi, 2048)
    assert abs(mu - ref) <= 1e-11 * max(1.0, abs(ref)), (mu, ref)
    mom = np.zeros((ND, N_PL + 1, 17))      # the same sums as the nodes' moments, without a handle
    mom[:, :, 0] = R / ND
    mom_dev, mu_dev = torch.tensor(mom, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    sq.sq_fermi_level_noalloc(mom_dev.data_ptr(), ND, N_PL, lo, hi, KT, inst["n_e"], 2048,
                              torch.cuda.current_stream().cuda_stream, mu_dev.data_ptr())
    assert abs(float(mu_dev) - ref) <= 1e-11 * max(1.0, abs(ref))
