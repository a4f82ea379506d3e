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


def _needle():
    xyz, tri = M.cylinder(0.5, 2.0, 7, 9)
    return np.ascontiguousarray(xyz * np.array([1e-5, 1e-5, 1.0])), tri


BODIES = {
    "needle": _needle,  # two axes whose grid steps are 1e-5 of the third's
    "plate": lambda: M.plate(1.0),  # one axis without extent
    "satellite": lambda: M.satellite(2_000),
    "cavity": lambda: M.hemisphere_shell(1.0, 6, 18),
    "off centre": lambda: (M.icosphere(2, 0.25)[0] + np.array([40.0, -7.0, 3.0]), M.icosphere(2, 0.25)[1]),
}


# control volumes from tight to far beyond float's digits at a grid step
@pytest.mark.parametrize("wide", [1.02, 30.0, 1e5])
@pytest.mark.parametrize("body", list(BODIES))
def test_fp64_hits_do_not_depend_on_the_box_arithmetic(T, body, wide):
    xyz, tri = BODIES[body]()
    centre, radius = M.bounding_sphere(xyz)
    # (hits fall with the square of the width: the farthest volumes mostly check that none is lost or added)
    N = 40_000 if wide < 2 else 200_000
    kw = dict(**W.base_state(S=7.0), dir=(0.2, 0.3, -1.0), eps_diffuse=0.9, A_ref=1.0, max_bounces=32, seed=17,
              r_cv=radius * wide, center=tuple(centre), precision=1)
    got = []
    for width in (2, 8):
        c = T.tpmc_create(0)
        try:
            T.tpmc_set_launch(c, block=0, bvh_width=width)
            mesh = T.tpmc_mesh_load(c, xyz, tri)
            assert T.tpmc_mesh_info(c, mesh)["bvh_width"] == width
            got.append(T.tpmc_trace(c, mesh, T.make_params(**kw), N))
        finally:
            T.tpmc_destroy(c)
    assert [got[0][k] for k in KEYS] == [got[1][k] for k in KEYS]
    if wide < 2 and body != "needle":
        assert got[0]["n_hits"] > 500
