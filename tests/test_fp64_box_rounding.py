"""FP64 launches on binary trees test boxes in float: the same arithmetic on the CPU, against the boxes in double.

The builder's grid and paddings (bvh.cpp) and the kernel's slab test (make_ray, box_start, ray_to_grid, trav_inner of
trace.cuh) are restated in numpy, rounding by rounding; the hardware reciprocal, good to one unit in the last place, is
taken one unit high, one low and exact.  A ray that passes through a triangle's box, as double has it, must pass the
float test, also when the closest hit so far is the point in the box that the ray goes for.
"""
import numpy as np
import pytest

F, D = np.float32, np.float64
BIG = D(2.0 ** 23)


def _down(v):
    f = v.astype(F)
    return np.where(f.astype(D) > v, np.nextafter(f, F(-np.inf)), f).astype(D)


def _up(v):
    f = v.astype(F)
    return np.where(f.astype(D) < v, np.nextafter(f, F(np.inf)), f).astype(D)


def _padded(lo, hi, scale):
    return _down(lo - (1e-5 * scale + 4e-7 * np.abs(lo))), _up(hi + (1e-5 * scale + 4e-7 * np.abs(hi)))


def _grid(lo, hi, scale):
    a, b = _padded(lo, hi, scale)
    step = 2.0 ** np.ceil(np.log2(np.maximum(b - a, 1e-30) / 65533.0))
    step = np.where(65533.0 * step < b - a, 2 * step, step)
    return _down(a - step), step


def _fma(a, b, c):
    """float fma: the product of two floats is exact in double."""
    return (a.astype(D) * b.astype(D) + c.astype(D)).astype(F)


def _float_test(o, d, t0, tlo, qlo, qhi, origin, step, tbest, ulps):
    inv = (F(1.0) / d.astype(F)).astype(F)
    for _ in range(abs(ulps)):
        inv = np.nextafter(inv, F(np.inf) * F(np.sign(ulps))).astype(F)
    sa = (step.astype(F) * inv).astype(F)
    g = ((t0[:, None] * d + o) - origin) / step
    oi = ((g + BIG) * sa.astype(D)).astype(F)
    lo_first = sa >= 0
    near = (BIG + np.where(lo_first, qlo, qhi)).astype(F)
    far = (BIG + np.where(lo_first, qhi, qlo)).astype(F)
    tn, tf = _fma(near, sa, -oi), _fma(far, sa, -oi)
    rel = (tlo - t0).astype(F)
    tnear = (rel - F(1e-6) * np.abs(rel)).astype(F)
    cull = tbest - t0
    with np.errstate(invalid="ignore"):
        cull = _up(cull + 1e-6 * np.abs(cull)).astype(F)
    tmin = np.maximum(tn.max(axis=1), tnear)
    tmax = np.minimum(tf.min(axis=1), cull)
    tmax = np.where(np.isinf(tmax), tmax, _fma(np.abs(tmax), np.full_like(tmax, 1e-6), tmax))
    return tmin <= tmax


def _box_start(o, d, centre, radius):
    x, y = (o - centre.astype(F).astype(D)).astype(F), d.astype(F)
    od, dd = (x * y).sum(axis=1, dtype=F), (y * y).sum(axis=1, dtype=F)
    t = (-od / dd - F(1.001) * F(radius) / np.sqrt(dd)).astype(F)
    t0 = (t - F(1e-4) * np.abs(t)).astype(F)
    return np.where((t0 > 0) & (t0 < 1e30), t0, 0).astype(D)


@pytest.mark.parametrize("ulps", [-1, 0, 1])
@pytest.mark.parametrize("centre", [(0.0, 0.0, 0.0), (40.0, -7.0, 3.0), (3e4, 2e4, -1e4)])
@pytest.mark.parametrize("extent", [(1, 1, 1), (1, 1, 0), (1e-3, 1e-3, 1), (1e-5, 1e-5, 1), (1, 1e-4, 1e-2)])
def test_float_boxes_reject_no_box_that_the_ray_meets(extent, centre, ulps):
    rng = np.random.default_rng(11)
    n = 30_000
    extent, centre = np.array(extent, D), np.array(centre, D)
    lo, hi = centre - extent / 2, centre + extent / 2
    radius = np.sqrt(((hi - lo) ** 2).sum()) / 2
    origin, step = _grid(lo, hi, radius)
    # boxes of all sizes inside the mesh, and a point in each: inside, on faces, on edges, at corners
    size = extent * np.exp(rng.uniform(np.log(1e-6), 0.0, (n, 3)))
    blo = lo + (extent - size) * rng.uniform(size=(n, 3))
    bhi = np.minimum(blo + size, hi)
    w = rng.uniform(size=(n, 3))
    w = np.where(rng.uniform(size=(n, 3)) < 0.5, np.round(w), w)
    point = blo + (bhi - blo) * w
    # directions of all slopes; starts from the surface to 1e5 radii away
    d = rng.normal(size=(n, 3)) * np.exp(rng.uniform(np.log(1e-6), 0.0, (n, 3))) * 50.0
    speed = np.sqrt((d * d).sum(axis=1))
    back = radius * np.exp(rng.uniform(np.log(1e-7), np.log(1e5), n)) / speed
    o = point - back[:, None] * d
    tlo = 1e-9 / speed
    t_in = ((point - o) * d).sum(axis=1) / speed ** 2  # where the ray, as rounded, is next to the point
    pass_tri = t_in > tlo
    a, b = _padded(blo, bhi, radius)
    qlo = np.clip(np.floor((a - origin) / step) - 1.0, 0, 65535)
    qhi = np.clip(np.ceil((b - origin) / step) + 1.0, 0, 65535)
    for seeded in (True, False):
        # a seeded ray's distances count from before the mesh's bounding sphere, a re-emitted one's from its start
        t0 = _box_start(o, d, centre, radius) if seeded else np.zeros(n)
        use = pass_tri if seeded else pass_tri & (back * speed < 2 * radius)
        assert use.sum() > 10_000
        for tbest in (np.full(n, np.inf), t_in):
            ok = _float_test(o, d, t0, tlo, qlo, qhi, origin, step, tbest, ulps)
            assert bool(ok[use].all()), (seeded, int((use & ~ok).sum()))
