"""Gauss density over column counts either side of where a warp takes more than one column's tridiagonal
(608 columns; the cells have 640, padding nodes included, and 512), one Krylov step and many, FP64.

Tolerance 1e-10 relative: the QL iteration is backward stable, about k 2^-53 of the spectrum's width, and
a weight moves by that over the gap of its node; the sums over k nodes of every column average it."""
import numpy as np
import pytest

from oracle import gauss_sq
from workloads import tiny_instance

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(9, 8, 8), (8, 8, 9), (7, 7, 8)])
@pytest.mark.parametrize("k", [1, 2, 31])
def test_density_over_column_counts(n, k):
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq
    inst = tiny_instance(seed=51, n=n, h=(0.8, 0.75, 0.7), n_atoms=4, n_o=2, r_cut=1.7, n_pl=8)
    ref = gauss_sq.run(inst, k=k)
    h = sq.sq_setup(sq.Desc(inst, sq.SQ_FP64, bounds=(-5.0, 60.0)))
    try:
        mu, rho, eb = sq.sq_gauss_density(h, k, int(np.prod(n)))
    finally:
        sq.sq_destroy(h)
    assert abs(mu - ref["mu"]) <= 1e-10 * max(1.0, abs(ref["mu"]))
    assert np.abs(rho - ref["rho"]).max() <= 1e-10 * np.abs(ref["rho"]).max()
    assert abs(eb - ref["E_band"]) <= 1e-10 * max(1.0, abs(ref["E_band"]))
