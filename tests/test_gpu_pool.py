"""Particles seeded into the pool against particles seeded inside the trace kernel, and the front boxes, on the GPU.

A counting launch (tpmc_set_counters) always seeds inside the trace kernel, so it is the reference for the pool: the
sums are integers over the same particles, so they are compared bit for bit.
"""
import numpy as np
import pytest

from tpmc_inputs import meshes as M
from tpmc_inputs import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("sum_dv_q", "sum_rdv_q", "n_particles", "n_hits", "n_hit_particles", "n_truncated", "CD_sigma", "status")


@pytest.fixture(scope="module")
def T():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1312_3691_gb300.build import build

    build()
    from paper_1312_3691_gb300 import tpmc

    return tpmc


def _base(T, **kw):
    return T.make_params(**{**W.base_state(S=6.0), "dir": (0.3, -0.2, 1.0), "eps_diffuse": 0.9, "A_ref": 1.0,
                            "max_bounces": 64, "seed": 99, **kw})


# (items, particles each): the pool's smallest launches, of several items and of one; several items a batch with ragged ends; over two
# batches of 2^26 (both streams, and the first pool again); many items inside one segment of 256 work indices
@pytest.mark.parametrize("K,N", [(2, (1 << 21) + 5), (1, (1 << 22) + 3), (1, 6 << 20), (1, (1 << 23) + 1), (3, 12_000_017), (7, 25_000_003),
                                 (400_000, 97)])
@pytest.mark.parametrize("width", [2, 4, 8])
@pytest.mark.parametrize("gsi", ["maxwell", "cll"])
def test_pool_gives_the_fused_sums(T, K, N, width, gsi):
    xyz, tri = M.satellite(3_000)
    kw = dict(gsi_model=T.TPMC_GSI_CLL, alpha_n=0.9, sigma_t=0.8) if gsi == "cll" else {}
    dirs = np.random.default_rng(1).normal(size=(K, 3))
    c = T.tpmc_create(0)
    try:
        T.tpmc_set_launch(c, block=0, bvh_width=width)
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        import torch

        d = torch.from_numpy(dirs).cuda()

        def swept(counting):
            T.tpmc_set_counters(c, counting)
            out = torch.zeros(K * T.RESULT_BYTES // 8, dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()
            T.tpmc_sweep_device(c, mesh, _base(T, **kw), d, None, K, N, out)
            torch.cuda.synchronize()
            rows = out.view(K, -1).cpu()
            return torch.cat([rows[:, :35], rows[:, 39:]], dim=1)  # all but the work counters, the id and ms

        pooled, fused = swept(False), swept(True)
        assert T.tpmc_memory_info(c)["used"] > K * N * 32 or K * N > 1 << 25  # the pool was there
        assert bool((pooled == fused).all())
        assert bool((pooled[:, 31] == N).all())  # n_particles: 25 doubles and six sums before it
    finally:
        T.tpmc_destroy(c)


# lengths of segments, from 64 work indices on: powers of two up to 2,048 behind rough rays (the satellite), 1,024
# without (the cylinder in a tight control volume); ragged ends in each
@pytest.mark.parametrize("N", [(1 << 23) + 2047, 12_000_001, 23_000_003, 47_000_033, (1 << 26) + 1])
@pytest.mark.parametrize("body", ["satellite", "cylinder"])
def test_segment_lengths(T, body, N):
    xyz, tri = M.satellite(3_000) if body == "satellite" else M.cylinder(0.5, 2.0, 24, 5)
    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        p = _base(T, r_cv=1.01 * float(np.sqrt((xyz ** 2).sum(axis=1).max())))
        pooled = T.tpmc_trace(c, mesh, p, N)
        T.tpmc_set_counters(c, True)
        fused = T.tpmc_trace(c, mesh, p, N)
        assert pooled["n_particles"] == N
        assert {k: pooled[k] for k in KEYS} == {k: fused[k] for k in KEYS}
    finally:
        T.tpmc_destroy(c)


@pytest.mark.parametrize("cv", ["tight", "wide", "box", "maxwell box"])
@pytest.mark.parametrize("body", ["satellite", "cylinder", "plate"])
def test_rough_rays_drop_no_particle_that_hits(T, body, cv):
    """S over its whole range (rough rays are not used above 15.9), 1e6 particles each, in control volumes that make
    most particles miss (rough rays first) or not: the fused kernel, which seeds every particle exactly, as reference."""
    xyz, tri = {"satellite": lambda: M.satellite(3_000), "cylinder": lambda: M.cylinder(0.5, 2.0, 24, 5),
                "plate": lambda: M.plate(1.0)}[body]()
    S = np.array([0.01, 0.1, 0.35, 0.7, 1.0, 1.5, 2.0, 2.5, 2.8, 3.2, 3.9, 4.0, 5.0, 6.0, 7.0, 8.0, 9.5, 11.0, 13.0,
                  15.8, 15.9, 16.0, 25.0, 50.0])
    centre, radius = M.bounding_sphere(xyz)
    kw = dict(center=tuple(centre), r_cv=radius * (1.02 if cv == "tight" else 3.0))
    if "box" in cv:
        kw = dict(cv_kind=T.TPMC_CV_BOX_MAXWELL if "maxwell" in cv else T.TPMC_CV_BOX_FLUX,
                  box_lo=tuple(xyz.min(axis=0) - 3.0), box_hi=tuple(xyz.max(axis=0) + 4.0))
    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        dirs = np.random.default_rng(5).normal(size=(len(S), 3))
        got = []
        for counting in (False, True):
            T.tpmc_set_counters(c, counting)
            got.append(T.tpmc_sweep(c, mesh, _base(T, **kw), dirs, S, 1_000_000))
        for pooled, fused in zip(*got):
            assert [pooled[k] for k in KEYS] == [fused[k] for k in KEYS]
    finally:
        T.tpmc_destroy(c)


@pytest.mark.parametrize("budget_mib", [24, 80, 300, 1200, 2048])
def test_pool_yields_to_the_memory_budget(T, budget_mib):
    """A pool of any size gives the same sums; meshes loaded after it find the room they would have had."""
    xyz, tri = M.cylinder(0.5, 2.0, 32, 7)
    N = (1 << 25) + 4097
    c = T.tpmc_create(0, budget_mib << 20)
    try:
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        r = T.tpmc_trace(c, mesh, _base(T), N)
        assert T.tpmc_memory_info(c)["used"] <= budget_mib << 20
        T.tpmc_set_counters(c, True)
        f = T.tpmc_trace(c, mesh, _base(T), N)
        assert [r[k] for k in KEYS] == [f[k] for k in KEYS]
        big = M.satellite(60_000)  # 16 MB on the device
        extra = [T.tpmc_mesh_load(c, *big) for _ in range(1 if budget_mib < 80 else 3)]
        T.tpmc_set_counters(c, False)
        again = T.tpmc_trace(c, mesh, _base(T), N)
        assert [again[k] for k in KEYS] == [f[k] for k in KEYS]
        assert len(extra) > 0
    finally:
        T.tpmc_destroy(c)


# r_cv: spheres from tight to 80 bodies wide; long: flux boxes close around the body and as many metres long upstream,
# at S = 50, so that rays that hit start beyond the front boxes' reach (256 to 512 extents for binary trees, 8 radii for
# wide ones) as well as within it
@pytest.mark.parametrize("r_cv,long", [(0.75, 0), (40.0, 0), (0, 6), (0, 1000)])
@pytest.mark.parametrize("name", ["plate", "cylinder"])
@pytest.mark.parametrize("width", [2, 8])
def test_front_rejects_no_particle_that_hits(T, orc, name, r_cv, long, width):
    """Control volumes from tight to beyond the front boxes' reach: the oracle's hits."""
    xyz, tri = M.plate(1.0) if name == "plate" else M.cylinder(0.3, 0.8, 12, 2)
    # aim: particles are seeded on the far volume, so the flow is cold and few of them meet the body
    N = 20_000 if 0 < r_cv < 1 else 1_000_000
    kw = dict(eps_diffuse=0.9, A_ref=1.0, max_bounces=16, seed=3)
    if long:
        lo, hi = xyz.min(axis=0) - 0.05, xyz.max(axis=0) + 0.05
        hi[2] += long
        kw.update(W.base_state(S=50.0), dir=(0.0, 0.0, -1.0), cv_kind=T.TPMC_CV_BOX_FLUX, box_lo=tuple(lo), box_hi=tuple(hi))
    else:
        kw.update(W.base_state(S=8.0), dir=(0.02, 0.01, -1.0), r_cv=r_cv)
    c = T.tpmc_create(0)
    try:
        T.tpmc_set_launch(c, block=0, bvh_width=width)
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        r = T.tpmc_trace(c, mesh, T.make_params(**kw), N)
    finally:
        T.tpmc_destroy(c)
    o, _, rec = orc.trace(orc.Mesh(xyz, tri), orc.make_params(**kw), N, records=True, K=1)
    assert r["n_particles"] == N
    # float positions are off by 6e-8 of the volume's size: particles that near to a silhouette edge may fall on either side
    edge = 8.0 * 6e-8 * (r_cv or long) / 0.5 * max(1.0, float(o["n_hits"]))
    assert abs(int(r["n_hits"]) - int(o["n_hits"])) <= 2 + edge, (r["n_hits"], o["n_hits"])
    assert o["n_hits"] >= 50
    if long:
        assert int(((rec["n_hits"] > 0) & (rec["pos"][:, 2] > 0.5 * long)).sum()) >= 10
    if 0 < r_cv < 1:
        assert r["n_hits"] > 1000 and abs(r["CD"] - o["CD"]) <= 1e-4 * abs(o["CD"]) + 3 * o["CD_sigma"]


def test_empty_mesh_counts_every_particle(T):
    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, np.zeros((0, 3)), np.zeros((0, 3), np.uint32))
        for N in (1, 33, (1 << 25) + 5):
            r = T.tpmc_trace(c, mesh, _base(T, r_cv=1.0), N)
            assert r["n_particles"] == N and r["n_hits"] == 0 and r["CD"] == 0.0
    finally:
        T.tpmc_destroy(c)


@pytest.mark.parametrize("budget_mib", [96, 700, 2500, 0])
def test_served_large_queries_match_direct_calls(T, budget_mib):
    """Served queries large enough for the steps' pools, among small ones and direct calls that use the context's own
    pool and make the others give their memory back: every result as alone."""
    bodies = [M.cylinder(0.5, 2.0, 32, 7), M.satellite(3_000)]
    sizes = [(0, (1 << 23) + 1), (1, 30_000_001), (0, 100_003), (1, (1 << 23) + 77), (1, 5_000_000), (0, 40_000_000)]
    c = T.tpmc_create(0, budget_mib << 20)
    try:
        meshes = [T.tpmc_mesh_load(c, *b) for b in bodies]
        params = [_base(T, stream_id=k, want_panels=k % 2 == 1) for k in range(len(sizes))]
        alone = []
        for (m, N), p in zip(sizes, params):
            r = T.tpmc_trace(c, meshes[m], p, N)
            if p.want_panels:
                r["panels"] = T.tpmc_panel_sums(c, r["query_id"], len(bodies[m][1]))
                T.tpmc_panels(c, r["query_id"], len(bodies[m][1]))
            alone.append(r)
        for _ in range(2):
            ids = [T.tpmc_submit(c, meshes[m], p, N) for (m, N), p in zip(sizes, params)]
            extra = T.tpmc_mesh_load(c, *M.satellite(60_000))
            direct = T.tpmc_trace(c, meshes[1], params[0], 20_000_000)
            T.tpmc_mesh_unload(c, extra)
            for i, a, (m, N) in zip(ids, alone, sizes):
                r = T.tpmc_poll(c, i)
                assert [r[k] for k in KEYS] == [a[k] for k in KEYS]
                if "panels" in a:
                    assert (T.tpmc_panel_sums(c, i, len(bodies[m][1])) == a["panels"]).all()
                    T.tpmc_panels(c, i, len(bodies[m][1]))
            assert direct["n_particles"] == 20_000_000
        if budget_mib:
            assert T.tpmc_memory_info(c)["used"] <= budget_mib << 20
    finally:
        T.tpmc_destroy(c)
