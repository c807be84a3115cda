"""Atoms clustered in a larger cell: the fullest brick meets several times the mean number of images. The mixed
step stays the split one (its tables are sized by what the bricks need together, which hardly depends on
where the atoms are), also when atoms that were spread out gather, and agrees with the scalar step (SQ_STEP_SMEM_ROWS
at a value the slabs just fit) on the same instance.

Tolerance 1e-4 of each moment slot's scale, as for the other instances of the split step: FP32 columns (2^-24 per
operation, n_pl steps of a bounded recurrence), the projections summed in different orders, amplified below
1e3 by the restricted grad grad at the node."""
import numpy as np
import pytest

from workloads import gaussian_veff, tiny_instance

pytestmark = pytest.mark.gpu

S = {"l": 0, "width": 0.5, "gamma": 1.0, "rcut": 2.0}
P = {"l": 1, "width": 0.5, "gamma": 0.5, "rcut": 2.0}


@pytest.fixture(scope="module")
def sq():
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq as mod
    return mod


def _instance(spread):
    """100 atoms on a (10, 9, 11) bohr cell, within 1 bohr of its centre or spread over it."""
    inst = tiny_instance(seed=41, n=(20, 18, 22), h=(0.5, 0.5, 0.5), n_atoms=100, n_o=3, r_cut=2.0, n_pl=6, proj=[S, P])
    u = np.random.Generator(np.random.PCG64(5)).uniform(-1.0, 1.0, (100, 3))
    L = np.asarray(inst["L"], dtype=float)
    inst["pos"] = np.mod(0.5 * L + (0.5 * L * u if spread else u), L)
    inst["v_eff"] = gaussian_veff(inst["L"], inst["n"], inst["pos"])
    return inst


def _moments(sq, h, inst):
    sq.sq_moments(h)
    return sq.sq_moments_copy(h, int(np.prod(inst["n"])), inst["n_pl"])


def _close(a, b):
    for k in range(a.shape[2]):
        scale = max(np.abs(b[:, :, k]).max(), 1e-3)
        assert np.abs(a[:, :, k] - b[:, :, k]).max() <= 1e-4 * scale, k


def test_cluster_takes_the_split_step(sq, monkeypatch):
    inst = _instance(False)
    out = []
    for env in (None, "0"):
        if env is not None:
            monkeypatch.setenv("SQ_STEP_SMEM_ROWS", env)
        h = sq.sq_setup(sq.Desc(inst, sq.SQ_MIXED))
        try:
            out.append((_moments(sq, h, inst), sq.sq_step_launch_counts(h)))
        finally:
            sq.sq_destroy(h)
    assert out[0][1][0] > 0 and out[0][1][1] == out[0][1][2] == 0
    assert out[1][1][0] == 0 and out[1][1][2] > 0
    _close(out[0][0], out[1][0])


def test_gathering_atoms_grow_the_tables(sq):
    """spread -> cluster -> spread on one handle and in a graph captured before: the tables are reallocated in
    between, and the graph must not use the old ones."""
    import torch
    spread, cluster = _instance(True), _instance(False)
    # a fresh handle's result per layout; the split step's sums have a fixed order: equal to the last bit
    ref = {}
    for name, inst in (("spread", spread), ("cluster", cluster)):
        h = sq.sq_setup(sq.Desc(inst, sq.SQ_MIXED))
        try:
            ref[name] = _moments(sq, h, inst)
        finally:
            sq.sq_destroy(h)
    st = torch.cuda.Stream()
    h = sq.sq_setup(sq.Desc(spread, sq.SQ_MIXED, stream=st.cuda_stream))
    batch = None
    nd, n_pl = int(np.prod(spread["n"])), spread["n_pl"]
    try:
        batch = sq.Batch([h])
        batch.run()
        assert np.array_equal(sq.sq_moments_copy(h, nd, n_pl), ref["spread"])
        sq.sq_update_atoms(h, cluster["pos"], cluster["v_eff"])
        assert np.array_equal(_moments(sq, h, cluster), ref["cluster"])
        sq.sq_update_atoms(h, spread["pos"], spread["v_eff"])
        batch.run()                                   # captured with the first tables
        assert np.array_equal(sq.sq_moments_copy(h, nd, n_pl), ref["spread"])
        sq.sq_update_atoms(h, cluster["pos"], cluster["v_eff"])
        batch.run()
        assert np.array_equal(sq.sq_moments_copy(h, nd, n_pl), ref["cluster"])
        c = sq.sq_step_launch_counts(h)
        assert c[0] > 0 and c[1] == c[2] == 0
    finally:
        if batch is not None:
            batch.close()
        sq.sq_destroy(h)
