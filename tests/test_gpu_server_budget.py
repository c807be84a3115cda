"""Device memory a handle asks for: what a server of a given budget held must stay accepted.

The FP64 sweep holds nine G fields per point where a W of three would do, the mixed one brick tables and partial
projections. Sizes of the workloads below that a budget was made for (bytes of the plan with three W fields and
without those tables) bound what a server must still take, in smaller waves if need be."""
import numpy as np
import pytest

from workloads import make_instance, tiny_instance


@pytest.fixture(scope="module")
def sq():
    from paper_2006_03697_gb300 import build
    build.build()
    from paper_2006_03697_gb300 import sq as mod
    return mod


def _small(atoms=2, n_o=4):
    return tiny_instance(seed=23, n=(11, 10, 12), h=(0.35, 0.35, 0.35), n_atoms=atoms, n_o=n_o, r_cut=2.5, n_pl=16)


def test_the_40_cube_workload_is_no_larger_than_before(sq):
    assert sq.sq_footprint_bytes(sq.Desc(make_instance(2), sq.SQ_MIXED)) <= 50.7e9


@pytest.mark.gpu
@pytest.mark.parametrize("precision,share", [("fp64", 0.5), ("mixed", 0.6), ("mixed", 0.8)])
def test_request_over_the_budget_runs_in_smaller_waves(sq, precision, share):
    """A budget below the usual plan's bytes but above the smallest plan's: the request is served, alone and as a
    trajectory of two snapshots, with the results of a handle of the usual plan (FP64 1e-10, mixed 1e-7: the
    tiles' columns do not depend on the waves, only sums over projections and nodes change their order)."""
    mode = sq.SQ_FP64 if precision == "fp64" else sq.SQ_MIXED
    tol = 1e-10 if precision == "fp64" else 1e-7
    inst = _small()
    moved = dict(inst, pos=np.asarray(inst["pos"]) + 0.07)
    descs = [sq.Desc(i, mode, bounds=(-8.0, 90.0)) for i in (inst, moved)]
    need = sq.sq_footprint_bytes(descs[0])
    srv = sq.Server(hbm_budget_bytes=int(share * need), max_inflight=2)
    got = []
    try:
        srv.submit(descs[0], tag=0)
        srv.submit(descs[0], tag=1, traj=1)
        srv.submit(descs[1], tag=2, traj=1)
        while len(got) < 3:
            got += srv.poll(timeout_ms=200)
    finally:
        srv.close()
    assert all(r["status"] == 0 for r in got), [(r["status"], r["error"]) for r in got]
    got = {r["tag"]: r for r in got}
    for tag, i in ((0, inst), (1, inst), (2, moved)):
        ref = sq.run(i, mode, bounds=(-8.0, 90.0))
        for k in ("E_band", "E_s", "E_nl", "F", "N_check"):
            assert abs(got[tag][k] - ref[k]) <= tol * max(1.0, abs(ref[k])), (tag, k)
        assert np.abs(got[tag]["sigma"] - ref["sigma"]).max() <= max(tol, 1e-9)
