"""The set-up kernel's two splits (few queries: table in blocks of its own; many: one block each) on the GPU."""
import math

import numpy as np
import pytest

from tpmc_inputs import meshes as M
from tpmc_inputs import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def T():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1312_3691_gb300.build import build

    build()
    from paper_1312_3691_gb300 import tpmc

    return tpmc


# S at the ends of its range, where the latitude law cancels, and where its lower tail is steep
@pytest.mark.parametrize("S", [0.01, 0.05, 0.35, 1.0, 2.0, 7.0, 16.0, 50.0])
@pytest.mark.parametrize("cv", ["sphere", "box"])
def test_both_splits_give_the_same_query(T, orc, S, cv):
    """64 queries in one sweep (one set-up block each) and each alone (split set-up): the same bits; the flux is the
    oracle's to 1e-13 (FP64 rounding of a dozen operations)."""
    xyz, tri = M.icosphere(1, 1.0)
    K, N = 64, 257
    rng = np.random.default_rng(3)
    dirs = rng.normal(size=(K, 3))
    dirs[:3] = [(0, 0, 1), (0, 0, -1), (1e-9, 0, 1)]  # the rotation's special cases
    kw = dict(**W.base_state(S=S), eps_diffuse=0.9, A_ref=math.pi, r_cv=1.5, max_bounces=8, seed=5)
    if cv == "box":
        kw.update(cv_kind=T.TPMC_CV_BOX_FLUX, box_lo=(-1.2, -1.1, -1.3), box_hi=(1.2, 1.4, 1.1))
    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        swept = T.tpmc_sweep(c, mesh, T.make_params(**kw, dir=(0, 0, 1)), dirs, np.full(K, S), N)
        for k in (0, 1, 2, 3, K - 1):
            alone = T.tpmc_sweep(c, mesh, T.make_params(**kw, dir=(0, 0, 1), stream_id=k), dirs[k:k + 1], [S], N)[0]
            for key in ("sum_dv_q", "sum_rdv_q", "n_hits", "CD", "CD_sigma", "force", "gamma", "fixed_quantum", "status"):
                assert alone[key] == swept[k][key], (k, key)
            assert alone["n_particles"] == N
        okw = {key: v for key, v in kw.items() if key != "cv_kind"}
        ores = orc.trace(orc.Mesh(xyz, tri), orc.make_params(**okw, dir=dirs[3], cv_kind=1 if cv == "box" else 0, stream=3), N)[0]
        assert abs(swept[3]["gamma"] / ores["gamma"] - 1) < 1e-13
    finally:
        T.tpmc_destroy(c)


def test_rejected_items_report_their_status(T):
    """A sweep's items with a speed ratio out of range are refused one by one, the others are as without them."""
    xyz, tri = M.icosphere(1, 1.0)
    S = np.array([7.0, 0.009, 51.0, 7.0])
    kw = dict(**W.base_state(S=7.0), dir=(0, 0, 1), eps_diffuse=1.0, A_ref=math.pi, r_cv=1.5, max_bounces=8, seed=5)
    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        r = T.tpmc_sweep(c, mesh, T.make_params(**kw), None, S, 1000)
        ok = T.tpmc_sweep(c, mesh, T.make_params(**kw), None, np.full(4, 7.0), 1000)
        assert [x["status"] for x in r] == [T.TPMC_OK, T.TPMC_EINVAL, T.TPMC_EINVAL, T.TPMC_OK]
        assert r[0]["sum_dv_q"] == ok[0]["sum_dv_q"] and r[3]["sum_dv_q"] == ok[3]["sum_dv_q"]
    finally:
        T.tpmc_destroy(c)


@pytest.mark.parametrize("offset", [0.0, 0.3])
def test_containment_at_its_limit(T, offset):
    """A control volume is accepted exactly when its radius exceeds the farthest vertex's distance."""
    xyz, tri = M.cylinder(0.4, 1.3, 9, 2)
    centre = np.array([offset, -offset, 0.1])
    far = np.sqrt(((xyz[np.unique(tri)] - centre) ** 2).sum(axis=1)).max()
    kw = dict(**W.base_state(S=7.0), dir=(0, 0, 1), eps_diffuse=1.0, A_ref=1.0, max_bounces=8, seed=5, center=tuple(centre))
    lo, hi = xyz.min(axis=0), xyz.max(axis=0)
    box = {k: v for k, v in kw.items() if k != "center"}
    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        for grow, ok in ((-1e-6, False), (-1e-12, False), (1e-12, True), (1e-6, True), (1.0, True)):
            params = [T.make_params(**kw, r_cv=far * (1 + grow)),
                      T.make_params(**box, cv_kind=T.TPMC_CV_BOX_FLUX, box_lo=tuple(lo - max(grow, 0)), box_hi=tuple(hi + grow))]
            for p in params:
                if ok:
                    assert T.tpmc_trace(c, mesh, p, 100)["n_particles"] == 100
                else:
                    with pytest.raises(T.TpmcError) as e:
                        T.tpmc_trace(c, mesh, p, 100)
                    assert e.value.status == T.TPMC_EINVAL
    finally:
        T.tpmc_destroy(c)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N", [1, 33, 4096, 20_000])
def test_calls_in_turn_read_their_own_set_up(T, precision, N):
    """Short calls one after another on one context, each with its own speed ratio, direction and seed, so with tables,
    items and sums that the next call's set-up writes over: each gives the bits it gives on a context of its own."""
    xyz, tri = M.icosphere(2, 1.0)
    base = dict(eps_diffuse=0.9, A_ref=math.pi, r_cv=1.5, max_bounces=8, precision=precision)
    calls = [dict(**W.base_state(S=S), **base, dir=d, seed=int(10 * S))
             for S, d in ((0.05, (0, 0, 1)), (50.0, (1, 0.2, 0)), (7.0, (-1, 2, 0.5)), (1.0, (0, -1, 0)))]
    keys = ("sum_dv_q", "sum_rdv_q", "n_hits", "n_hit_particles", "n_particles", "CD", "CD_sigma", "gamma")
    want = []
    for kw in calls:
        c = T.tpmc_create(0)
        try:
            mesh, p = T.tpmc_mesh_load(c, xyz, tri), T.make_params(**kw)
            rs = T.tpmc_trace(c, mesh, p, N), T.tpmc_sweep(c, mesh, p, np.array([kw["dir"]], float), None, N)[0]
            want.append([[r[k] for k in keys] for r in rs])
        finally:
            T.tpmc_destroy(c)
    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        params = [T.make_params(**kw) for kw in calls]
        for _ in range(25):
            for p, kw, w in zip(params, calls, want):
                r = T.tpmc_trace(c, mesh, p, N)
                assert [r[k] for k in keys] == w[0]
                r = T.tpmc_sweep_noalloc(c, mesh, p, np.array([kw["dir"]], float), None, N)[0]
                assert [r[k] for k in keys] == w[1]
    finally:
        T.tpmc_destroy(c)
