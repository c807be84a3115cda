"""Device Lanczos against the oracle's over the step counts where its kernels change shape: one step, a
few, either side of a warp's 32 lanes, and the largest. Ragged 5 x 6 x 7 cell, FP64.

Tolerance 1e-9 of the interval's width: Gram-Schmidt twice keeps the Krylov vectors orthogonal to
1e-15, so the tridiagonals agree to about k 1e-14 and the Ritz extremes with them."""
import pytest

from oracle import sq_oracle as orc
from workloads import tiny_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 3, 17, 31, 33, 128])
def test_bounds_over_step_counts(k):
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq
    inst = tiny_instance(seed=1, n=(5, 6, 7), h=(0.7, 0.65, 0.6), n_atoms=3, n_o=2, r_cut=2.0, n_pl=4)
    lo, hi = orc.lanczos_bounds(orc.Problem(inst), k)
    h = sq.sq_setup(sq.Desc(inst, sq.SQ_FP64, lanczos_k=k))
    try:
        sq.sq_moments(h)
        glo, ghi = sq.sq_get_bounds(h)
    finally:
        sq.sq_destroy(h)
    assert abs(glo - lo) <= 1e-9 * (hi - lo)
    assert abs(ghi - hi) <= 1e-9 * (hi - lo)
