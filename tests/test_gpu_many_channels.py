"""Handles that never run the split mixed step (FP64, or more than 4 projector channels per atom) list the images of
their windows only, not of whole bricks past the windows' edges: blocks that hold their projector rows in shared
memory must not lose it to rows nothing reads. Windows of 10 x 10 x 10 points here, bricks of 4; atom counts at
which the windows' rows just fit."""
import numpy as np
import pytest

from workloads import tiny_instance

pytestmark = pytest.mark.gpu

PROJ = [{"l": 0, "width": 0.5, "gamma": 1.0, "rcut": 2.0}, {"l": 1, "width": 0.5, "gamma": 0.5, "rcut": 2.0},
        {"l": 1, "width": 0.4, "gamma": 0.5, "rcut": 2.0}]


@pytest.mark.parametrize("precision,atoms", [("fp64", 26), ("mixed", 36)])
def test_projector_rows_stay_in_shared_memory(precision, atoms):
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq
    inst = tiny_instance(seed=3, n=(9, 8, 10), h=(0.4, 0.4, 0.4), n_atoms=atoms, n_o=2, r_cut=1.61, n_pl=2, kT=0.5, proj=PROJ)
    got = {}
    for mode in (sq.SQ_FP64, sq.SQ_FP64 if precision == "fp64" else sq.SQ_MIXED):
        h = sq.sq_setup(sq.Desc(inst, mode, bounds=(-30.0, 200.0)))
        try:
            sq.sq_moments(h)
            got[mode] = sq.sq_moments_copy(h, int(np.prod(inst["n"])), inst["n_pl"])
            counts = sq.sq_step_launch_counts(h)
        finally:
            sq.sq_destroy(h)
    assert counts[1] == inst["n_pl"] + 1 and counts[2] == 0, counts
    if precision == "mixed":     # FP32 columns: 2^-24 per operation, two steps
        a, b = got[sq.SQ_MIXED], got[sq.SQ_FP64]
        for k in range(a.shape[2]):
            assert np.abs(a[:, :, k] - b[:, :, k]).max() <= 1e-5 * max(np.abs(b[:, :, k]).max(), 1e-3), k
