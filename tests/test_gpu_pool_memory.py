"""Pools of seeded particles and the memory around them: who waits for it, how often it is taken, on the GPU."""
import time

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
    return T.make_params(**{**W.base_state(S=7.0), "dir": (0.3, -0.2, 1.0), "eps_diffuse": 0.9, "A_ref": 1.0,
                            "max_bounces": 64, "seed": 7, **kw})


def _room(T, c):
    i = T.tpmc_memory_info(c)
    return i["budget"] - i["used"]


def test_panel_query_waits_for_pool_memory_and_nobody_waits_with_it(T):
    """A served query whose panel loads find the budget taken by the pools of a running step is left queued until that
    step is over; submitting and polling (without a time-out) go on meanwhile, and the query is served in the end."""
    xyz, tri = M.satellite(60_000)
    budget = 4 << 30
    c = T.tpmc_create(0, budget)
    try:
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        for _ in range(2):  # the pools of both steps in flight
            for i in [T.tpmc_submit(c, mesh, _base(T), 1 << 24) for _ in range(2)]:
                T.tpmc_poll(c, i)
        p = _base(T, want_panels=True, stream_id=3)
        alone = T.tpmc_trace(c, mesh, p, 1000)
        panels = T.tpmc_panel_sums(c, alone["query_id"], len(tri))
        while _room(T, c) >= 24 * len(tri):  # panel loads nobody reads fill the rest
            T.tpmc_trace(c, mesh, p, 1000)
        t0 = time.perf_counter()
        # two steps in flight: queries are admitted again when the first is over, while the large one runs
        first, big = T.tpmc_submit(c, mesh, _base(T), 1_000_000_000), T.tpmc_submit(c, mesh, _base(T), 12_000_000_000)
        time.sleep(0.02)
        longest, waiting = 0.0, []
        while True:
            a = time.perf_counter()
            if len(waiting) < 4:
                waiting.append(T.tpmc_submit(c, mesh, p, 1000))
            done = T.tpmc_poll(c, big, 0)
            longest = max(longest, time.perf_counter() - a)
            if done is not None:
                break
            time.sleep(0.002)
        assert time.perf_counter() - t0 > 0.4  # the large query ran for long enough to tell
        assert longest < 0.1, longest
        assert T.tpmc_poll(c, first)["n_particles"] == 1_000_000_000
        for i in waiting:
            r = T.tpmc_poll(c, i)
            assert [r[k] for k in KEYS] == [alone[k] for k in KEYS]
            assert (T.tpmc_panel_sums(c, i, len(tri)) == panels).all()
        assert T.tpmc_memory_info(c)["used"] <= budget
        again = T.tpmc_submit(c, mesh, _base(T), (1 << 23) + 5)  # large queries are served as before
        assert T.tpmc_poll(c, again)["n_particles"] == (1 << 23) + 5
    finally:
        T.tpmc_destroy(c)


def test_rising_counts_take_a_pool_for_each_power_of_two(T):
    """Forty calls, each of 2^20 particles more than the last: the pool is taken for 2^24, 2^25 and 2^26 particles."""
    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, *M.plate(1.0))
        T.tpmc_trace(c, mesh, _base(T), 1000)
        before = T.tpmc_memory_info(c)["n_allocs"]
        for k in range(40):
            N = (1 << 24) - 5 + (k << 20)
            assert T.tpmc_trace(c, mesh, _base(T), N)["n_particles"] == N
        assert T.tpmc_memory_info(c)["n_allocs"] - before <= 3
    finally:
        T.tpmc_destroy(c)


def test_serving_takes_a_pool_for_each_step_in_flight_once(T):
    """Large queries of rising size, served smallest first: one allocation for each of the two steps."""
    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, *M.plate(1.0))
        T.tpmc_poll(c, T.tpmc_submit(c, mesh, _base(T), 1000))
        before = T.tpmc_memory_info(c)["n_allocs"]
        sizes = [(1 << 23) + 7 + (k << 21) for k in range(12)]
        ids = [T.tpmc_submit(c, mesh, _base(T), N) for N in sizes]
        assert [T.tpmc_poll(c, i)["n_particles"] for i in ids] == sizes
        assert T.tpmc_memory_info(c)["n_allocs"] - before <= 2
    finally:
        T.tpmc_destroy(c)


def test_device_sweep_of_thousands_of_batches_only_enqueues(T):
    """2^35 particles (on no mesh) with room for batches of 2^23: the call returns while most of them are to come, and
    every item counts its particles, those traced after the pool's batches as well."""
    import torch

    K, N = 64, 1 << 29
    c = T.tpmc_create(0, 1200 << 20)
    try:
        mesh = T.tpmc_mesh_load(c, np.zeros((0, 3)), np.zeros((0, 3), np.uint32))
        out = torch.zeros(K * T.RESULT_BYTES // 8, dtype=torch.int64, device="cuda")
        p = _base(T, r_cv=1.0)
        T.tpmc_sweep_device(c, mesh, p, None, None, K, 1 << 20, out)
        torch.cuda.synchronize()
        assert T.tpmc_memory_info(c)["used"] > 64 << 23  # the pool is there
        t0 = time.perf_counter()
        T.tpmc_sweep_device(c, mesh, p, None, None, K, N, out)
        enqueued = time.perf_counter() - t0
        torch.cuda.synchronize()
        whole = time.perf_counter() - t0
        # a host that waits for room in the queue is there to the last few thousand of 8,192 launches
        assert enqueued < 0.25 * whole, (enqueued, whole)
        assert bool((out.view(K, -1)[:, 31] == N).all())  # n_particles: 25 doubles and six sums before it
    finally:
        T.tpmc_destroy(c)


def test_what_follows_the_pool_gives_the_same_sums(T):
    """2^33 particles and some, with room for batches of 2^23: 896 of them go through the pool, 128 and a ragged rest do
    not; the sums are the fused launch's."""
    import torch

    K, N = 3, (1 << 33) // 3 + 12_345
    xyz, tri = M.plate(1.0)
    c = T.tpmc_create(0, 1200 << 20)
    try:
        mesh = T.tpmc_mesh_load(c, xyz, tri)
        rows = []
        for counting in (False, True):
            T.tpmc_set_counters(c, counting)
            out = torch.zeros(K * T.RESULT_BYTES // 8, dtype=torch.int64, device="cuda")
            d = torch.from_numpy(np.random.default_rng(2).normal(size=(K, 3))).cuda()
            torch.cuda.synchronize()
            T.tpmc_sweep_device(c, mesh, _base(T), d, None, K, N, out)
            torch.cuda.synchronize()
            got = out.view(K, -1).cpu()
            rows.append(torch.cat([got[:, :35], got[:, 39:]], dim=1))  # all but the work counters, the id and ms
        assert bool((rows[0] == rows[1]).all())
        assert bool((rows[0][:, 31] == N).all())
    finally:
        T.tpmc_destroy(c)


def test_pools_leave_the_device_to_others(T):
    """With 8 GB of the device free, a context whose budget allows more takes at most a quarter for its pools, each
    time; another user of the device finds what is left."""
    import torch

    c = T.tpmc_create(0)
    try:
        mesh = T.tpmc_mesh_load(c, *M.plate(1.0))
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        rest = 8 << 30
        if free < 2 * rest:
            pytest.skip("the device is in use")
        others = torch.empty(free - rest, dtype=torch.uint8, device="cuda")
        before = T.tpmc_memory_info(c)["used"]
        assert T.tpmc_trace(c, mesh, _base(T), 1 << 27)["n_particles"] == 1 << 27
        assert 0 < T.tpmc_memory_info(c)["used"] - before <= rest // 4 + (1 << 20)
        ids = [T.tpmc_submit(c, mesh, _base(T), 1 << 25) for _ in range(3)]
        assert [T.tpmc_poll(c, i)["n_particles"] for i in ids] == [1 << 25] * 3
        more = torch.empty(rest // 3, dtype=torch.uint8, device="cuda")
        del others, more
    finally:
        T.tpmc_destroy(c)
        torch.cuda.empty_cache()
