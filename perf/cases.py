"""The work that programs have this library do, as cases that can be timed.

A case names a mesh of tpmc_inputs, a free stream, a surface model, a particle
count and the entry point that a program calls.  listed() has twelve, from a
4,096-particle look at one attitude to the 3,072-attitude sweep; draw() gives
more of the same ranges.  prepare() loads the mesh into a context, as a program
does once; run() is the call a program repeats.

exact() is the same sums over the same Philox streams in 64 bits, written with
plain torch: inverse CDFs by bisection and Newton steps, closest hits by testing
every triangle.
"""
import functools
import math
import weakref

import numpy as np
import torch

from paper_1312_3691_gb300 import tpmc as T
from tpmc_inputs import meshes, workloads

EXACT_TESTS = 1.2e10  # ray/triangle pairs that exact() tests in a few seconds


def listed():
    base = dict(cv="sphere", gsi="maxwell", eps=1.0, precision="fp32", max_bounces=64, panels=False, attitudes=1)
    case = lambda name, **kw: dict(base, name=name, **kw)  # noqa: E731
    return [
        # the smallest call: a first look at one attitude (launches and latency only)
        case("quick_look", call="trace", mesh="sphere", size=1280, S=7.5, eps=0.9, particles=4096),
        # a control loop that may not allocate: eight candidate attitudes a tick
        case("control_tick", call="noalloc", mesh="cylinder", size=4096, S=7.0, eps=0.9, attitudes=8,
             particles=20_000),
        # verification in double precision: the icosphere benchmark
        case("sphere_fp64", call="trace", mesh="sphere", size=1280, S=7.5, precision="fp64", particles=100_000),
        # the other control volume and surface model: flux-weighted box, Cercignani-Lampis-Lord
        case("box_cll", call="trace", mesh="sphere", size=1280, S=5.0, cv="box", gsi="cll", particles=1_000_003),
        # the plate and cylinder sweeps (32 incidences x 3 speed ratios), 1e7 particles a case
        case("plate_sweep", call="sweep", mesh="plate", size=2, S=0.0, eps=0.0, attitudes=96, particles=10_000_000),
        case("cylinder_sweep", call="sweep", mesh="cylinder", size=4096, S=0.0, attitudes=96, particles=10_000_000),
        # a cavity: many bounces per particle
        case("hemisphere", call="trace", mesh="hemisphere", size=6048, S=40.0, max_bounces=200, particles=10_000_000),
        # one attitude of the concave satellite in detail: 1e8 particles, pressure and shear of every panel
        case("satellite_panels", call="trace", mesh="satellite", size=60_000, S=7.0, eps=0.9, panels=True,
             particles=100_000_000),
        # restoring moments over the incidence and roll grid at the flight conditions
        case("moments", call="sweep", mesh="satellite", size=60_000, S=8.47, attitudes=152, particles=262_144),
        # the attitude data base: 32 x 32 yaw and pitch x 3 speed ratios in one device-resident call
        case("attitude_sweep", call="sweep_device", mesh="satellite", size=60_000, S=0.0, eps=0.9, attitudes=3072,
             particles=1_048_576),
        # a finely meshed satellite
        case("satellite_500k", call="trace", mesh="satellite", size=500_000, S=7.0, eps=0.9, particles=10_000_000),
        # a burst of queries of mixed sizes and meshes through the serving loop
        case("serving_burst", call="serve", mesh="mixed", size=60_000, S=0.0, eps=0.9, attitudes=32,
             particles=100_000_000),
    ]


def draw(rng):
    """One more case: any mesh, entry point and option, sizes spread over their whole range."""
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    mesh = rng.choice(["sphere", "plate", "cylinder", "cylinder", "hemisphere", "satellite", "satellite"])
    size = {"sphere": 20 * 4 ** rng.randint(1, 4), "plate": 2, "cylinder": log(60, 20_000), "hemisphere": log(200, 12_000),
            "satellite": log(2_000, 120_000)}[mesh]
    call = rng.choice(["trace", "trace", "sweep", "sweep", "sweep_device", "noalloc", "serve"])
    precision = "fp64" if call == "trace" and rng.random() < 0.2 else "fp32"
    most = 300_000 if precision == "fp64" else 60_000_000 if mesh == "hemisphere" else 1_000_000_000
    attitudes = {"trace": 1, "sweep": log(2, 600), "sweep_device": log(2, 4000), "noalloc": log(1, 64),
                 "serve": log(2, 40)}[call]
    top = {"trace": 100_000_000, "serve": 30_000_000}.get(call, 10_000_000)
    particles = min(log(1_000, top), max(1, most // attitudes))
    return dict(call=call, mesh="mixed" if call == "serve" else mesh, size=size if call != "serve" else 60_000,
                S=round(rng.uniform(2.0, 12.0), 3), eps=rng.choice([0.0, 0.9, 1.0]), attitudes=attitudes,
                particles=particles, precision=precision, cv=rng.choice(["sphere", "sphere", "box"]),
                gsi=rng.choice(["maxwell", "maxwell", "cll"]), panels=call == "trace" and rng.random() < 0.3,
                max_bounces=64 if mesh != "hemisphere" else 200)


# ------------------------------------------------------------------ inputs
@functools.lru_cache(maxsize=8)
def _mesh(kind, size):
    if kind == "sphere":
        return meshes.icosphere(int(round(math.log(size / 20, 4))))
    if kind == "plate":
        return meshes.plate(1.0)
    if kind == "cylinder":  # 2 n (n_axial + 1) triangles with about eight azimuths per band
        if size == 4096:
            return meshes.cylinder(0.5, 2.0, 128, 15)
        az = max(5, int(round(math.sqrt(4 * size))))
        return meshes.cylinder(0.5, 2.0, az, max(1, int(round(size / (2 * az))) - 1))
    if kind == "hemisphere":  # n_lon (2 n_lat - 1) triangles
        if size == 6048:
            return meshes.hemisphere_shell(1.0, 32, 96)
        lat = max(2, int(round(math.sqrt(size / 6))))
        return meshes.hemisphere_shell(1.0, lat, 3 * lat)
    return meshes.satellite(size)


A_REF = dict(sphere=math.pi, plate=1.0, cylinder=2.0, hemisphere=math.pi, satellite=2.0)
QUANTITIES = ("force", "torque", "CD", "CD_sigma", "CF", "CM", "gamma", "weight")
WHOLE = ("sum_dv_q", "sum_rdv_q", "n_particles", "n_hits", "n_hit_particles", "n_truncated")


def _inputs(case, seed, kind):
    """(keyword arguments of make_params, directions [K, 3], speed ratios [K]) of a case on mesh `kind`."""
    rng = np.random.default_rng(seed)
    K, S = case["attitudes"], case["S"]
    if kind == "hemisphere":  # a hyperthermal stream along the cavity's axis
        state = workloads.hemisphere_case(S=S)["params"]
        state = {k: state[k] for k in ("n", "T_inf", "m", "V", "T_W")}
        dirs = np.array([(0.05, 0.0, 1.0)] * K) + 0.05 * rng.normal(size=(K, 3))
    else:
        state = workloads.base_state(S=S or 7.0)
        dirs = rng.normal(size=(K, 3))
        if case["call"] == "sweep" and kind in ("plate", "cylinder"):  # incidences of 0 to 90 degrees
            a = np.radians(90.0) * (np.arange(K) % 32 + rng.uniform(0.0, 1.0)) / 32
            dirs = np.stack([np.sin(a), 0.0 * a, -np.cos(a)], axis=1)
        elif case["call"] == "sweep":
            state = workloads.table1_state()
            a = np.radians(np.arange(K) % 19 * 10.0 - 90.0 + rng.uniform(0.0, 10.0))
            b = np.radians(22.5 * (np.arange(K) // 19))
            dirs = -np.stack([np.sin(a) * np.cos(b), np.sin(a) * np.sin(b), np.cos(a)], axis=1)
    ratios = np.full(K, S) if S else np.array([2.0, 5.0, 10.0])[np.arange(K) * 3 // K]
    if not S and kind == "satellite":
        ratios = np.array([5.0, 7.5, 10.0])[np.arange(K) * 3 // K]
    xyz, tri = _mesh(kind, case["size"])
    centre, radius = meshes.bounding_sphere(xyz)
    kw = dict(state, eps_diffuse=case["eps"], A_ref=A_REF[kind], max_bounces=case["max_bounces"],
              seed=int(rng.integers(1, 1 << 62)), stream_id=int(rng.integers(0, 1 << 20)), r_cv=1.05 * radius,
              center=tuple(centre), ref_point=(0.0, 0.0, 0.1), l_ref=2.0, want_panels=case["panels"],
              precision=T.TPMC_FP64 if case["precision"] == "fp64" else T.TPMC_FP32)
    if case["cv"] == "box":
        lo, hi = xyz.min(axis=0), xyz.max(axis=0)
        kw.update(cv_kind=T.TPMC_CV_BOX_FLUX, box_lo=tuple(lo - 0.2), box_hi=tuple(hi + 0.2))
    if case["gsi"] == "cll":
        kw.update(gsi_model=T.TPMC_GSI_CLL, alpha_n=0.9, sigma_t=0.8)
    return kw, dirs / np.linalg.norm(dirs, axis=1, keepdims=True), ratios


@functools.lru_cache(maxsize=1)
def _stream():
    return torch.cuda.Stream()


class State:
    def __init__(self, case, seed):
        self.case = case
        self.ctx = T.tpmc_create(0)
        self._gone = weakref.finalize(self, T.tpmc_destroy, self.ctx)
        if case["call"] == "serve":
            rng = np.random.default_rng(seed)
            kinds = [("sphere", 1280), ("cylinder", 4096), ("satellite", case["size"])]
            ids = [T.tpmc_mesh_load(self.ctx, *_mesh(*k)) for k in kinds]
            self.queries = []
            # counts spaced evenly in their logarithm, in random order: every seed has the same work
            counts = np.exp(np.linspace(math.log(min(1e5, case["particles"])), math.log(case["particles"]), case["attitudes"]))
            for n, i in zip(rng.permutation(counts), rng.permutation(np.arange(case["attitudes"]) % 3)):
                one = dict(case, call="trace", attitudes=1, size=kinds[i][1], S=case["S"] or float(rng.uniform(3.0, 12.0)))
                kw, dirs, _ = _inputs(one, int(rng.integers(1 << 40)), kinds[i][0])
                self.queries.append((ids[i], T.make_params(**kw, dir=dirs[0]), int(n)))
            return
        kind = case["mesh"]
        xyz, tri = _mesh(kind, case["size"])
        self.n_tri = len(tri)
        self.mesh = T.tpmc_mesh_load(self.ctx, xyz, tri)
        kw, self.dirs, self.S = _inputs(case, seed, kind)
        self.params = T.make_params(**kw, dir=self.dirs[0])
        if case["call"] == "sweep_device":
            T.tpmc_set_stream(self.ctx, _stream())
            self.d_dirs = torch.from_numpy(self.dirs).cuda()
            self.d_S = torch.from_numpy(self.S).cuda()
            self.d_out = torch.zeros(case["attitudes"] * T.RESULT_BYTES // 8, dtype=torch.int64, device="cuda")
            torch.cuda.synchronize()


def prepare(case, seed):
    return State(case, seed)


def _gathered(results):
    out = {k: np.array([r[k] for r in results], dtype=np.float64) for k in QUANTITIES}
    out.update({k: np.array([r[k] for r in results], dtype=np.int64) for k in WHOLE})
    return out


def run(s):
    case, N = s.case, s.case["particles"]
    if case["call"] == "trace":
        r = T.tpmc_trace(s.ctx, s.mesh, s.params, N)
        out = _gathered([r])
        if case["panels"]:
            out["pressure"], out["shear"] = T.tpmc_panels(s.ctx, r["query_id"], s.n_tri)
        return out
    if case["call"] == "sweep":
        return _gathered(T.tpmc_sweep(s.ctx, s.mesh, s.params, s.dirs, s.S, N))
    if case["call"] == "noalloc":
        return _gathered(T.tpmc_sweep_noalloc(s.ctx, s.mesh, s.params, s.dirs, s.S, N))
    if case["call"] == "sweep_device":
        T.tpmc_sweep_device(s.ctx, s.mesh, s.params, s.d_dirs, s.d_S, case["attitudes"], N, s.d_out)
        rows = s.d_out.view(case["attitudes"], -1)
        # the result record: 25 doubles (force to fixed_quantum), then 12 sums and counts
        return {"values": rows.view(torch.float64)[:, :25], "counts": rows[:, 25:37]}
    ids = [T.tpmc_submit(s.ctx, *q) for q in s.queries]
    return _gathered([T.tpmc_poll(s.ctx, i) for i in ids])


# --------------------------------------------------------------------- work
def _particles(case):
    if case["call"] != "serve":
        return case["particles"] * case["attitudes"]
    lo, hi, K = math.log(min(1e5, case["particles"])), math.log(case["particles"]), case["attitudes"]
    return sum(math.exp(lo + (hi - lo) * k / max(1, K - 1)) for k in range(K))


def work(case):
    """Seeding (150 flops), the root box (20); for a particle that hits (about 0.2, 2 in a cavity) the boxes down to
    one leaf (40 each), one triangle test (35) and the re-emission (30).  Bytes: the mesh and the queries read, the
    results and panel loads written."""
    n, tri = _particles(case), case["size"]
    hits = {"plate": 0.3, "sphere": 0.8, "cylinder": 0.5, "hemisphere": 2.0}.get(case["mesh"], 0.2)
    flops = n * (170.0 + hits * (40.0 * math.log2(max(2, tri)) + 65.0))
    bytes_ = 36.0 * tri + case["attitudes"] * (300.0 + T.RESULT_BYTES) + (16.0 * tri if case["panels"] else 0.0)
    return {"bytes": bytes_, "flops": flops}


# -------------------------------------------------- the same sums in 64 bits
_SQRT_PI = math.sqrt(math.pi)


def _philox(pid, stream, block, seed):
    """Philox4x32-10 words of counters (pid, stream, block), as int64 tensors below 2^32."""
    mask = 0xFFFFFFFF
    c = [pid & mask, pid >> 32, torch.full_like(pid, stream), torch.full_like(pid, block)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # wraps modulo 2^64: the low 32 bits and the next 32 are right
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _uniform(w):
    return ((w >> 9).double() + 0.5) * 2.0 ** -23


def _latitude(u, S):
    """x = sin(latitude) with H(x) = u."""
    D = math.exp(-S * S) + _SQRT_PI * (1 + 2 * S * S) * math.erf(S) / (2 * S)

    def cdf(x):
        a = S * x
        return (_SQRT_PI / (4 * S) * (2 * a * a + 1) * torch.special.erfc(-a) + 0.5 * x * torch.exp(-a * a)
                - (_SQRT_PI / (4 * S) * (2 * S * S + 1) * math.erfc(S) - 0.5 * math.exp(-S * S))) / D

    grid = torch.linspace(-1, 1, 4097, dtype=torch.float64, device=u.device)
    at = cdf(grid)
    i = torch.searchsorted(at, u).clamp_(1, 4096)
    lo, hi = grid[i - 1], grid[i]
    x = lo + (hi - lo) * ((u - at[i - 1]) / (at[i] - at[i - 1])).clamp_(0, 1)
    for _ in range(5):
        a = S * x
        step = (cdf(x) - u) * D / (torch.exp(-a * a) + _SQRT_PI * a * torch.special.erfc(-a))
        x = torch.minimum(torch.maximum(x - torch.nan_to_num(step), lo), hi)
    return x


def _normal_speed(u, s):
    """x > 0 of density 2 x exp(-(x - s)^2) / Z with distribution function u."""
    q = 1.0 - u
    es = _SQRT_PI * s
    neg = s < 0
    Z = torch.where(neg, 1.0 + es * torch.special.erfcx(s.abs()), torch.exp(-s * s) + es * torch.special.erfc(-s))

    def tail(x):
        y = x - s
        e = torch.where(neg, torch.exp(-x * (x - 2 * s)), torch.exp(-y * y))
        upper = torch.where(neg, e * (1.0 + es * torch.special.erfcx(torch.where(neg, y, 1.0))), e + es * torch.special.erfc(y))
        return upper / Z, 2 * x * e / Z

    lo, hi = torch.zeros_like(s), s.clamp(min=0) + 6.5
    for _ in range(14):
        x = 0.5 * (lo + hi)
        above = tail(x)[0] > q
        lo, hi = torch.where(above, x, lo), torch.where(above, hi, x)
    x = 0.5 * (lo + hi)
    for _ in range(4):
        Q, p = tail(x)
        x = torch.minimum(torch.maximum(x + torch.nan_to_num((Q - q) / p), lo), hi)
    return x


def _flux(s):
    return (math.exp(-s * s) + _SQRT_PI * s * math.erfc(-s)) / (2 * _SQRT_PI)


def _seeded(pid, kw, d, S, N):
    """Positions and velocities (c_mp units) of particles `pid`, and the flux into the volume over n c."""
    w = _philox(pid, kw["stream_id"], 0, kw["seed"])
    angle = ((((w[0] & 0x1FF) | ((w[1] & 0x1FF) << 9) | ((w[2] & 0x1F) << 18)).double()) + 0.5) * 2.0 ** -23 * (2 * math.pi)
    u = [_uniform(x) for x in w]
    r = torch.sqrt(-torch.log(u[3]))
    t1, t2 = r * torch.cos(angle), r * torch.sin(angle)
    if "box_lo" in kw:
        lo, hi = np.array(kw["box_lo"]), np.array(kw["box_hi"])
        ext, flux = hi - lo, []
        speed = [float(S * (-d[f // 2] if f % 2 == 0 else d[f // 2])) for f in range(6)]
        for f in range(6):
            flux.append(float(ext[(f // 2 + 1) % 3] * ext[(f // 2 + 2) % 3]) * _flux(speed[f]))
        cum, ends = 0.0, []
        for f in range(5):
            cum += flux[f] / sum(flux)
            ends.append(math.floor(N * cum))
        face = torch.bucketize(pid, torch.tensor(ends, device=pid.device), right=True)
        vn = _normal_speed(u[2], torch.tensor(speed, dtype=torch.float64, device=pid.device)[face])
        pos, vel = [], []
        for i in range(3):
            on, first = face // 2 == i, (face // 2 + 1) % 3 == i
            high = face % 2 == 0
            free = float(lo[i]) + torch.where(first, u[0], u[1]) * float(ext[i])
            pos.append(torch.where(on, torch.where(high, float(hi[i]), float(lo[i])), free))
            vel.append(torch.where(on, torch.where(high, -vn, vn), S * float(d[i]) + torch.where(first, t1, t2)))
        return torch.stack(pos, 1), torch.stack(vel, 1), sum(flux)
    x = _latitude(u[0], S)
    c = torch.sqrt((1 - x) * (1 + x))
    ct, st = torch.cos(2 * math.pi * u[1]), torch.sin(2 * math.pi * u[1])
    vn = _normal_speed(u[2], S * x)
    t1 = S * c + t1
    pos = torch.stack([c * ct, c * st, -x], 1)
    vel = torch.stack([-vn * c * ct + t1 * x * ct + t2 * st, -vn * c * st + t1 * x * st - t2 * ct, vn * x + t1 * c], 1)
    # Rodrigues rotation of +z onto d about z x d
    k = np.array([-d[1], d[0], 0.0])
    sin, cos = np.linalg.norm(k), float(d[2])
    if sin < 1e-12:
        R = np.diag([1.0, math.copysign(1.0, cos), math.copysign(1.0, cos)])
    else:
        k = k / sin
        X = np.array([[0, -k[2], k[1]], [k[2], 0, -k[0]], [-k[1], k[0], 0]])
        R = np.eye(3) + sin * X + (1 - cos) * (X @ X)
    R = torch.from_numpy(R).to(pid.device)
    centre = torch.tensor(kw["center"], dtype=torch.float64, device=pid.device)
    into = kw["r_cv"] ** 2 * (_SQRT_PI * math.exp(-S * S) + (math.pi / (2 * S) + math.pi * S) * math.erf(S))
    return centre + kw["r_cv"] * pos @ R.T, vel @ R.T, into


def _closest(o, v, tris, last, near):
    """Distance (in |v|) and index of the first triangle that the rays meet; index -1 where there is none."""
    A, e1, e2 = tris
    best, at = torch.full_like(o[:, 0], math.inf), torch.full_like(last, -1)
    for lo in range(0, len(A), 4096):
        a, b, c = A[lo:lo + 4096], e1[lo:lo + 4096], e2[lo:lo + 4096]
        for p in range(0, len(o), 4_000_000 // len(a) + 1):
            n = slice(p, p + 4_000_000 // len(a) + 1)
            d, r = v[n, None, :], o[n, None, :] - a
            h = torch.linalg.cross(d, c[None], dim=2)
            det = (h * b).sum(2)
            f = 1.0 / det
            s = f * (r * h).sum(2)
            q = torch.linalg.cross(r, b[None].expand_as(r), dim=2)
            w = f * (q * d).sum(2)
            t = f * (q * c).sum(2)
            ok = (det != 0) & (s >= 0) & (w >= 0) & (s + w <= 1) & (t > near[n, None])
            ok &= torch.arange(lo, lo + len(a), device=o.device)[None] != last[n, None]
            t, i = torch.where(ok, t, math.inf).min(1)
            nearer = t < best[n]
            best[n], at[n] = torch.where(nearer, t, best[n]), torch.where(nearer, i + lo, at[n])
    return best, at


def _one(case, kw, xyz, tri, d, S):
    """The result of one query, in 64 bits."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    P = torch.from_numpy(xyz).to(dev)[torch.from_numpy(tri.astype(np.int64)).to(dev)]
    e1, e2 = P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]
    normal = torch.nn.functional.normalize(torch.linalg.cross(e1, e2, dim=1), dim=1)
    first = torch.nn.functional.normalize(e1, dim=1)
    second = torch.linalg.cross(normal, first, dim=1)
    N, cw = case["particles"], math.sqrt(kw["T_W"] / kw["T_inf"])
    ref = torch.tensor(kw["ref_point"], dtype=torch.float64, device=dev)
    vhat = torch.from_numpy(np.asarray(d)).to(dev)
    dv, rdv, squares = (torch.zeros(k, dtype=torch.float64, device=dev) for k in (3, 3, 1))
    shortest = 1e-9 if case["precision"] == "fp64" else 1e-6
    for at in range(0, N, 4_000_000):
        pid = torch.arange(at, min(N, at + 4_000_000), device=dev)
        o, v, into = _seeded(pid, kw, d, S, N)
        last = torch.full_like(pid, -1)
        drag = torch.zeros(len(pid), dtype=torch.float64, device=dev)
        row = torch.arange(len(pid), device=dev)
        for bounce in range(case["max_bounces"]):
            t, i = _closest(o, v, (P[:, 0].contiguous(), e1, e2), last, shortest / v.norm(dim=1))
            keep = i >= 0
            if not bool(keep.any()):
                break
            row, pid, o, v, last, t = (x[keep] for x in (row, pid, o, v, i, t))
            o = o + t[:, None] * v
            n, a, b = normal[last], first[last], second[last]
            u = _philox(pid, kw["stream_id"], 2 + bounce, kw["seed"])
            vn = (v * n).sum(1)
            sgn = torch.where(vn < 0, 1.0, -1.0).double()
            if "alpha_n" in kw:
                at_ = kw["sigma_t"] * (2 - kw["sigma_t"])
                r = torch.sqrt(-kw["alpha_n"] * torch.log(_uniform(u[0])))
                m = math.sqrt(1 - kw["alpha_n"]) * (-sgn * vn) / cw
                vn2 = torch.sqrt((r * r + m * m + 2 * r * m * torch.cos(2 * math.pi * _uniform(u[1]))).clamp(min=0))
                rho, phi = torch.sqrt(-at_ * torch.log(_uniform(u[2]))), 2 * math.pi * _uniform(u[3])
                keep_t = math.sqrt(1 - at_) / cw
                new = cw * ((sgn * vn2)[:, None] * n + (keep_t * (v * a).sum(1) + rho * torch.cos(phi))[:, None] * a
                            + (keep_t * (v * b).sum(1) + rho * torch.sin(phi))[:, None] * b)
            else:
                diffuse = (u[0] >> 9) < math.ceil(kw["eps_diffuse"] * 2 ** 23 - 0.5)
                out = cw * torch.sqrt(-torch.log(_uniform(u[1])))
                side, phi = cw * torch.sqrt(-torch.log(_uniform(u[2]))), 2 * math.pi * _uniform(u[3])
                new = ((sgn * out)[:, None] * n + (side * torch.cos(phi))[:, None] * a + (side * torch.sin(phi))[:, None] * b)
                new = torch.where(diffuse[:, None], new, v - 2 * vn[:, None] * n)
            change = v - new
            dv += change.sum(0)
            rdv += torch.linalg.cross(o - ref, change, dim=1).sum(0)
            drag.index_add_(0, row, change @ vhat)
            v = new
        squares += (drag * drag).sum()
    c = math.sqrt(2 * workloads.K_B * kw["T_inf"] / kw["m"])
    V = S * c
    gamma, q_inf = into * kw["n"] * c, 0.5 * kw["n"] * kw["m"] * V * V
    dv, rdv = dv.cpu().numpy(), rdv.cpu().numpy()
    force, torque = (gamma / N * kw["m"] * c * x for x in (dv, rdv))
    mean = float(dv @ d) / N
    var = max(0.0, (float(squares) - N * mean * mean) / max(1, N - 1))
    return dict(force=force, torque=torque, CD=float(force @ d) / (q_inf * kw["A_ref"]),
                CD_sigma=gamma * kw["m"] * c / (q_inf * kw["A_ref"]) * math.sqrt(var / N), CF=force / (q_inf * kw["A_ref"]),
                CM=torque / (q_inf * kw["A_ref"] * kw["l_ref"]), gamma=gamma, weight=gamma / N)


def exact(case, seed):
    if case["call"] in ("serve", "sweep_device") or case["panels"] or case["mesh"] == "hemisphere" \
            or float(_particles(case)) * case["size"] > EXACT_TESTS or case["attitudes"] > 400:
        return None
    kw, dirs, ratios = _inputs(case, seed, case["mesh"])
    xyz, tri = _mesh(case["mesh"], case["size"])
    c = math.sqrt(2 * workloads.K_B * kw["T_inf"] / kw["m"])
    rows = []
    for k in range(case["attitudes"]):
        S = kw["V"] / c if case["call"] == "trace" else float(ratios[k])
        rows.append(_one(case, dict(kw, stream_id=kw["stream_id"] + k), xyz, tri, dirs[k], S))
    out = {q: np.array([r[q] for r in rows], dtype=np.float64) for q in QUANTITIES}
    out.update({q: None for q in WHOLE})
    return out
