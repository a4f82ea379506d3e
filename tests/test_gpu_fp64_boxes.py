"""FP64 launches on binary trees test boxes in float, on 8-wide trees in double: the closest hits are the same."""
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


def _needle(thin):
    xyz, tri = M.cylinder(0.5, 2.0, 7, 9)
    return np.ascontiguousarray(xyz * np.array([thin, thin, 1.0])), tri


BODIES = {
    "needle": lambda: _needle(1e-5),  # two axes whose grid steps are 1e-5 of the third's
    "thin": lambda: _needle(1e-3),
    "plate": lambda: M.plate(1.0),  # one axis without extent
    "satellite": lambda: M.satellite(2_000),
    "cavity": lambda: M.hemisphere_shell(1.0, 6, 18),
    "off centre": lambda: (M.icosphere(2, 0.25)[0] + np.array([40.0, -7.0, 3.0]), M.icosphere(2, 0.25)[1]),
}


def _by_width(T, xyz, tri, kw, N, K):
    """Results and, with K > 0, records of the same launch on a binary and on an 8-wide tree."""
    got = []
    for width in (2, 8):
        c = T.tpmc_create(0)
        try:
            T.tpmc_set_launch(c, block=0, bvh_width=width)
            mesh = T.tpmc_mesh_load(c, xyz, tri)
            assert T.tpmc_mesh_info(c, mesh)["bvh_width"] == width
            p = T.make_params(**kw, precision=1)
            got.append((T.tpmc_trace(c, mesh, p, N), T.tpmc_trace_records(c, mesh, p, N, K=K)[1] if K else None))
        finally:
            T.tpmc_destroy(c)
    assert [got[0][0][k] for k in KEYS] == [got[1][0][k] for k in KEYS]
    return got


# Control volumes from tight to 30 bodies wide.  Of N particles N A_proj / (pi r_cv^2) hit, at least 100 of these
# 2,000,000 in the wide ones; the thin bodies, which next to none would meet, have the long volumes below.
@pytest.mark.parametrize("wide,N,least", [(1.02, 40_000, 500), (30.0, 2_000_000, 100)])
@pytest.mark.parametrize("body", ["plate", "satellite", "cavity", "off centre"])
def test_fp64_hits_do_not_depend_on_the_box_arithmetic(T, body, wide, N, least):
    xyz, tri = BODIES[body]()
    centre, radius = M.bounding_sphere(xyz)
    kw = dict(**W.base_state(S=7.0), dir=(0.2, 0.3, -1.0), eps_diffuse=0.9, A_ref=1.0, max_bounces=32, seed=17,
              r_cv=radius * wide, center=tuple(centre))
    got = _by_width(T, xyz, tri, kw, N, 0)
    assert got[0][0]["n_hit_particles"] >= least


@pytest.mark.parametrize("bodies", [3.0, 100.0, 1000.0])
@pytest.mark.parametrize("body", list(BODIES))
def test_fp64_hits_from_far_upstream(T, body, bodies):
    """A flux box close around the body across the stream and `bodies` of its narrower widths long against it, S = 50:
    hits whose rays start thousands of grid steps of the finest axis away, in number, particle by particle."""
    xyz, tri = BODIES[body]()
    lo, hi = xyz.min(axis=0), xyz.max(axis=0)
    axis = 0 if body in ("needle", "thin") else 2  # across the long body; along z for the others
    width = min(float(hi[a] - lo[a]) for a in range(3) if a != axis)
    length = bodies * width
    margin = 0.05 * (hi - lo)
    margin[axis] = 0.05 * width
    lo, hi = lo - margin, hi + margin
    hi[axis] += length
    flow = [0.0, 0.0, 0.0]
    flow[axis] = -1.0
    kw = dict(**W.base_state(S=50.0), dir=tuple(flow), eps_diffuse=0.9, A_ref=1.0, max_bounces=32, seed=23,
              cv_kind=T.TPMC_CV_BOX_FLUX, box_lo=tuple(lo), box_hi=tuple(hi))
    N = 2_000_000
    (res, a), (_, b) = _by_width(T, xyz, tri, kw, N, 4)
    for k in ("n_hits", "tri", "truncated"):
        assert (a[k] == b[k]).all()
    # of the particles from the far face, erf(25 / bodies) squared or more meet the body's cross section, and 1 in
    # 1 + 0.023 bodies starts there; those that start within half the length are not counted
    far = (a["n_hits"] > 0) & (a["pos"][:, axis] > hi[axis] - 0.5 * length)
    assert int(far.sum()) >= 50, int(far.sum())
    assert res["n_hit_particles"] >= 1000
