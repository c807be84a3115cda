"""Mixed precision where hundreds of projector rows meet a brick (many atoms and periodic images in a small cell):
the tensor-core sums must stay as close to FP64 as FP32 arithmetic comes, whatever their length.

Bar: 1e-6 relative on every energy against its own magnitude, as for the other mixed instances; 3e-6 Ha/bohr^3 on the
stress (n_pl = 12 steps of FP32 columns, 2^-24 per operation, times the restricted grad grad, below 1e2 here)."""
import numpy as np
import pytest

from workloads import tiny_instance

pytestmark = pytest.mark.gpu

S = {"l": 0, "width": 0.5, "gamma": 1.0, "rcut": 3.0}
P = {"l": 1, "width": 0.5, "gamma": 0.5, "rcut": 3.0}


@pytest.fixture(scope="module")
def sq():
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq as mod
    return mod


@pytest.mark.parametrize("atoms,bounds", [(12, (-30.0, 200.0)), (19, (-40.0, 300.0))])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_dense_cell_against_fp64(sq, atoms, bounds, seed):
    inst = tiny_instance(seed=seed, n=(6, 2, 3), h=(0.45, 0.45, 0.5), n_atoms=atoms, n_o=3, r_cut=2.3, n_pl=12, kT=0.5,
                         proj=[S, P])
    ref, got = (sq.run(inst, p, bounds=bounds) for p in (sq.SQ_FP64, sq.SQ_MIXED))
    for k in ("E_band", "E_s", "E_nl", "F"):
        assert abs(got[k] - ref[k]) <= 1e-6 * abs(ref[k]), (k, got[k], ref[k])
    assert np.abs(got["sigma"] - ref["sigma"]).max() <= 3e-6
