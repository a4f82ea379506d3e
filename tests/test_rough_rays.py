"""How far the rough rays of the seeding (may_hit) are off, emulated in double precision over samples of the uniforms.

The set-up widens the front boxes by 1.5 times what these bounds allow; a ray that is further off than the bounds
could be dropped although it hits.  The samples hold the 2,000 uniforms nearest 0 and 1 and tens of thousands between.
"""
import numpy as np
import pytest
import torch

K_H, Z_LO, Z_HI = 128, -5.5, 5.5
N_S, N_Z, S_LO, STEP = 193, 89, -8.0, 0.125
SQRT_PI = np.sqrt(np.pi)


def _uniforms():
    rng = np.random.default_rng(0)
    top = 2 ** 23 - 1
    near = np.arange(2000)
    spread = np.exp(rng.uniform(0, np.log(top), 20_000)).astype(np.int64)
    k = np.unique(np.concatenate([near, top - near, spread, top - spread, rng.integers(0, top, 20_000)]))
    return torch.from_numpy((k + 0.5) / 2 ** 23)


def _phi(z):
    return 0.5 * torch.special.erfc(-z / np.sqrt(2.0))


def _rough_quantile(u):
    p = torch.minimum(u, 1 - u)
    t = torch.sqrt(-2 * torch.log(p))
    z = t - (2.515517 + 0.802853 * t + 0.010328 * t * t) / (1 + 1.432788 * t + 0.189269 * t * t + 0.001308 * t ** 3)
    return torch.where(u < 0.5, -z, z)


def _root(cdf, u, lo, hi):
    """cdf(x) = u by bisection."""
    for _ in range(60):
        x = 0.5 * (lo + hi)
        below = cdf(x) < u
        lo, hi = torch.where(below, x, lo), torch.where(below, hi, x)
    return 0.5 * (lo + hi)


def _interpolated(tab, f, n):
    j = torch.clamp(torch.floor(f), 0, n - 2).long()
    w = torch.clamp(f - j, 0, 1)
    return (1 - w) * tab[j] + w * tab[j + 1]


def test_rough_quantile_bound():
    u = _uniforms()
    assert float((_rough_quantile(u) - torch.special.ndtri(u)).abs().max()) <= 4.5e-4


@pytest.mark.parametrize("S", [0.01, 0.1, 0.35, 1.0, 2.0, 2.5, 2.8, 3.2, 3.5, 3.9, 4.0, 4.5, 7.0, 10.0, 15.9])
def test_rough_latitude_bound(S):
    """The latitude is off by at most 1.7e-3 radians (S < 4), 4.5e-4 above."""
    s = torch.tensor(S, dtype=torch.float64)
    D = torch.exp(-s * s) + SQRT_PI * (1 + 2 * S * S) * torch.erf(s) / (2 * S)
    K1 = SQRT_PI / (4 * S) * (2 * S * S + 1) * torch.erfc(s) - 0.5 * torch.exp(-s * s)

    def cdf(x):
        a = S * x
        return (SQRT_PI / (4 * S) * (2 * a * a + 1) * torch.special.erfc(-a) + 0.5 * x * torch.exp(-a * a) - K1) / D

    def solve(u):
        return _root(cdf, u, -torch.ones_like(u), torch.ones_like(u))

    u = _uniforms()
    tab = solve(_phi(Z_LO + (Z_HI - Z_LO) * torch.arange(K_H + 1, dtype=torch.float64) / K_H))
    x = solve(u)
    rough = _interpolated(tab, (_rough_quantile(u) - Z_LO) / ((Z_HI - Z_LO) / K_H), K_H + 1)
    angle = lambda v: torch.atan2(torch.sqrt(torch.clamp((1 - v) * (1 + v), min=0)), v)  # noqa: E731
    assert float((angle(rough) - angle(x)).abs().max()) <= (1.7e-3 if S < 4 else 4.5e-4)


@pytest.mark.parametrize("lo,hi", [(-7.9, -4), (-4, -2), (-2, -1), (-1, 0), (0, 1), (1, 3), (3, 8), (8, 15.9)])
def test_rough_normal_speed_bound(lo, hi):
    """The normal speed is off by at most 2e-3 c_mp."""
    def cdf(s):
        neg = s < 0
        Z = torch.where(neg, 1 + SQRT_PI * s * torch.special.erfcx(s.abs()), torch.exp(-s * s) + SQRT_PI * s * torch.special.erfc(-s))

        def f(x):
            y = x - s
            e = torch.where(neg, torch.exp(-x * (x - 2 * s)), torch.exp(-y * y))
            up = torch.where(neg, e * (1 + SQRT_PI * s * torch.special.erfcx(torch.where(neg, y, torch.ones_like(y)))),
                             e + SQRT_PI * s * torch.special.erfc(y))
            return 1 - up / Z
        return f

    def solve(u, s):
        return _root(cdf(s), u, torch.zeros_like(s), s.clamp(min=0) + 12)

    u = _uniforms()
    s = torch.from_numpy(np.random.default_rng(1).uniform(lo, hi, len(u)))
    zs = Z_LO + STEP * torch.arange(N_Z, dtype=torch.float64)
    rows = torch.arange(int((lo - S_LO) / STEP), min(N_S - 1, int((hi - S_LO) / STEP) + 1) + 1)
    grid_s = (S_LO + STEP * rows.double())[:, None].expand(-1, N_Z).reshape(-1)
    tab = solve(_phi(zs).repeat(len(rows)), grid_s).reshape(len(rows), N_Z)
    x = solve(u, s)
    fs = (s - S_LO) / STEP - int(rows[0])
    i = torch.clamp(torch.floor(fs), 0, len(rows) - 2).long()
    a = torch.clamp(fs - i, 0, 1)
    fz = (_rough_quantile(u) - Z_LO) / STEP
    j = torch.clamp(torch.floor(fz), 0, N_Z - 2).long()
    b = torch.clamp(fz - j, 0, 1)
    rough = (1 - a) * ((1 - b) * tab[i, j] + b * tab[i, j + 1]) + a * ((1 - b) * tab[i + 1, j] + b * tab[i + 1, j + 1])
    assert float((rough - x).abs().max()) <= 2e-3
