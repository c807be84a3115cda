"""Device Lanczos against the oracle's over the channel counts where its H application changes kernel: one
channel, up to four (three, four, species with one and four), more than four. FP64, ragged 5 x 6 x 7 cell.

Tolerance 1e-9 of the interval's width: Gram-Schmidt twice keeps the Krylov vectors orthogonal to
1e-15, so the tridiagonals agree to about k 1e-14 and the Ritz extremes with them."""
import numpy as np
import pytest

from oracle import sq_oracle as orc
from workloads import tiny_instance

pytestmark = pytest.mark.gpu

S = {"l": 0, "width": 0.5, "gamma": 1.0, "rcut": 3.5}
P = {"l": 1, "width": 0.5, "gamma": 0.5, "rcut": 3.5}
S2 = {"l": 0, "width": 0.7, "gamma": -0.4, "rcut": 2.8}
P2 = {"l": 1, "width": 0.6, "gamma": -0.3, "rcut": 3.0}


@pytest.mark.parametrize("proj", [[[S]], [[P]], [[S, P]], [[S, P], [S2]], [[S, P, S2]], [[S], [S, P, S2, P2]]],
                         ids=["1", "3", "4", "4_and_1", "5", "1_and_8"])
def test_bounds_over_channel_counts(proj):
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq
    inst = tiny_instance(seed=3, n=(5, 6, 7), h=(0.7, 0.65, 0.6), n_atoms=3, n_o=2, r_cut=2.0, n_pl=4, proj=proj[0])
    inst["proj"] = proj
    inst["species"] = np.array([0, 1, 1]) % len(proj)
    lo, hi = orc.lanczos_bounds(orc.Problem(inst), 20)
    h = sq.sq_setup(sq.Desc(inst, sq.SQ_FP64, lanczos_k=20))
    try:
        sq.sq_moments(h)
        glo, ghi = sq.sq_get_bounds(h)
    finally:
        sq.sq_destroy(h)
    assert abs(glo - lo) <= 1e-9 * (hi - lo)
    assert abs(ghi - hi) <= 1e-9 * (hi - lo)
