"""The Fermi search (Newton steps on ln N inside a bracket, one cluster of blocks) against plain
bisection in NumPy on the same node sums, over dilute to nearly full bands, cold to hot smearing and
several Chebyshev-Gauss point counts (odd, below one point per thread, several per thread).

Tolerance: both stop on a bracket of 1e-13 max(1, |mu|); N(mu) itself carries M rounding errors of
1e-16 N, which move the root by about 1e-15 N / N'(mu) <= 1e-14 kT / (1 - filling): 1e-11 covers both."""
import numpy as np
import pytest

from workloads import tiny_instance

pytestmark = pytest.mark.gpu


def _bisect(R, lo, hi, kT, n_e, M):
    k = np.arange(M) + 0.5
    F = np.cos(np.outer(np.pi * k / M, np.arange(len(R)))) @ np.concatenate([[0.5 * R[0]], R[1:]])
    lam = 0.5 * (lo + hi) + 0.5 * (hi - lo) * np.cos(np.pi * k / M)

    def count(mu):
        x = (lam - mu) / kT
        e = np.exp(-np.abs(x))
        return 4.0 / M * np.sum(np.where(x > 0, e / (1 + e), 1 / (1 + e)) * F)

    a, b = lo - 40 * kT, hi + 40 * kT
    for _ in range(200):
        m = 0.5 * (a + b)
        a, b = (m, b) if count(m) < n_e else (a, m)
        if b - a < 1e-13 * max(1.0, abs(m)):
            break
    return 0.5 * (a + b)


@pytest.mark.parametrize("kT", [0.05, 3.17])
@pytest.mark.parametrize("filling", [0.003, 0.4, 0.97])
@pytest.mark.parametrize("M", [101, 2048, 6144])
def test_fermi_search_matches_bisection(kT, filling, M):
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq
    inst = tiny_instance(seed=21, n=(4, 4, 3), h=(0.7, 0.7, 0.7), n_atoms=1, n_o=1, r_cut=0.8, n_pl=24, kT=kT, M=M)
    nd = 48
    inst["n_e"] = 2 * nd * filling
    bounds = (-6.0, 12.0)
    rng = np.random.default_rng(5)
    x = rng.uniform(-0.9, 0.9, 400)      # node sums of a spectrum inside the interval
    R = nd * np.cos(np.outer(np.arange(25), np.arccos(x))).mean(axis=1)
    h = sq.sq_setup(sq.Desc(inst, sq.SQ_FP64, bounds=bounds))
    try:
        lo, hi = sq.sq_get_bounds(h)
        mu = sq.sq_fermi_level_sums(h, R)
    finally:
        sq.sq_destroy(h)
    ref = _bisect(R, lo, hi, kT, inst["n_e"], M)
    assert abs(mu - ref) <= 1e-11 * max(1.0, abs(ref)), (mu, ref)
