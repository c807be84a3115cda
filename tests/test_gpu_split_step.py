"""The split mixed step (stencil, projector apply and projections as kernels of their own) against the
scalar step with its projections in global memory (SQ_STEP_SMEM_ROWS=0) on the same instance, at the sizes
where the split kernels change shape: one to four projector channels per atom and two species
with different counts, waves of one and a few tiles (bricks shared by part of their tiles), ragged
cells, more projector rows in a brick than one pass holds, every stencil order, and windows wide enough for
the stencil's second variant.

Tolerance 1e-4 of each moment slot's scale: both paths hold FP32 columns (2^-24 per operation, n_pl steps of
a bounded recurrence) and sum the projections in different orders; the restricted grad grad at the node
amplifies that rounding by the ratio of the second-derivative weights to the result, below 1e3 here."""
import numpy as np
import pytest

from workloads import tiny_instance

pytestmark = pytest.mark.gpu

S = {"l": 0, "width": 0.5, "gamma": 1.0, "rcut": 3.5}
P = {"l": 1, "width": 0.5, "gamma": 0.5, "rcut": 3.5}
S2 = {"l": 0, "width": 0.7, "gamma": -0.4, "rcut": 2.8}
BASE = dict(seed=31, n=(5, 6, 7), h=(0.6, 0.55, 0.5), n_atoms=3, n_o=3, r_cut=2.6, n_pl=8)
CASES = {
    "one_channel": (dict(BASE, proj=[S]), 0),
    "two_channels": (dict(BASE, proj=[S, S2]), 0),
    "three_channels": (dict(BASE, proj=[P]), 0),
    "four_channels": (dict(BASE, proj=[S, P]), 0),
    "species_mix": (dict(BASE, proj=[S, P]), 0),
    "waves_of_1": (dict(BASE), 1),
    "waves_of_5": (dict(BASE), 5),
    "waves_of_13": (dict(BASE), 13),
    "dense_passes": (dict(BASE, n=(4, 4, 5), n_atoms=9), 0),
    "no1": (dict(BASE, n_o=1), 0),
    "no6": (dict(BASE, n_o=6), 0),
    "wide_window": (dict(seed=32, n=(2, 1, 2), h=(0.5, 0.9, 0.9), n_atoms=1, n_o=6, r_cut=21.2, n_pl=3), 0),
}


def _moments(sq, inst, wave):
    nd = int(np.prod(inst["n"]))
    h = sq.sq_setup(sq.Desc(inst, sq.SQ_MIXED, bounds=(-8.0, 60.0)))
    try:
        if wave:
            sq.sq_tune_step(h, 0, wave, 0)
        sq.sq_moments(h)
        return sq.sq_moments_copy(h, nd, inst["n_pl"]), sq.sq_step_launch_counts(h)
    finally:
        sq.sq_destroy(h)


@pytest.mark.parametrize("name", sorted(CASES))
def test_split_step_matches_global_projections(monkeypatch, name):
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq
    kw, wave = CASES[name]
    inst = tiny_instance(**kw)
    if name == "species_mix":
        inst["proj"] = [[S, P], [S2]]
        inst["species"] = np.array([0, 1, 1])
    a, ca = _moments(sq, inst, wave)
    assert ca[0] > 0 and ca[1] == ca[2] == ca[3] == 0
    monkeypatch.setenv("SQ_STEP_SMEM_ROWS", "0")
    b, cb = _moments(sq, inst, wave)
    assert cb[0] == 0 and cb[2] > 0
    for k in range(a.shape[2]):
        scale = max(np.abs(b[:, :, k]).max(), 1e-3)
        assert np.abs(a[:, :, k] - b[:, :, k]).max() <= 1e-4 * scale, k
