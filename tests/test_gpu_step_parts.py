"""The FP64 step with a block per brick and a warp per brick plane (waves of few bricks) against one block per
slab: waves from one tile to either side of the brick count where the rule changes, with the default and
with given warps per block, one and four projector channels.

Tolerance 1e-12 of each moment slot's scale: the same FP64 sums in another order (2^-53 per operation, n_pl
steps of a bounded recurrence), amplified by the restricted grad grad at the node by less than 1e3."""
import numpy as np
import pytest

from workloads import tiny_instance

pytestmark = pytest.mark.gpu

S = {"l": 0, "width": 0.5, "gamma": 1.0, "rcut": 3.5}
P = {"l": 1, "width": 0.5, "gamma": 0.5, "rcut": 3.5}


def _moments(sq, inst, warps, wave):
    h = sq.sq_setup(sq.Desc(inst, sq.SQ_FP64, bounds=(-8.0, 60.0)))
    try:
        sq.sq_tune_step(h, warps, wave, 0)
        sq.sq_moments(h)
        return sq.sq_moments_copy(h, int(np.prod(inst["n"])), inst["n_pl"])
    finally:
        sq.sq_destroy(h)


@pytest.mark.parametrize("proj", [[S], [S, P]], ids=["one_channel", "four_channels"])
@pytest.mark.parametrize("warps,wave", [(0, 1), (0, 3), (0, 20), (0, 27), (1, 1), (8, 2)])
def test_split_slabs_match_whole_slabs(proj, warps, wave):
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq
    # 80 tiles of 27 bricks in waves of 1, 3, 20, 27 and 2 tiles, against one wave; the rule changes at 608 bricks
    inst = tiny_instance(seed=41, n=(7, 8, 9), h=(0.6, 0.55, 0.5), n_atoms=3, n_o=2, r_cut=2.4, n_pl=6, proj=proj)
    a, b = _moments(sq, inst, warps, wave), _moments(sq, inst, 0, 0)
    for k in range(a.shape[2]):
        scale = max(np.abs(b[:, :, k]).max(), 1e-3)
        assert np.abs(a[:, :, k] - b[:, :, k]).max() <= 1e-12 * scale, k
