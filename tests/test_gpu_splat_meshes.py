"""The splat's kernels by the size of the mesh: with four and six view slots a
lane, units of two points below 50,000 and 150,000 triangles and of four from
there on. Sampling and the views looked at equal the oracle's on either side, and
the walk of segments (a low lane limit) gives the pooled passes' keys."""
from dataclasses import replace

import numpy as np
import pytest

import oracle as O
from paper_2601_19901_gb300 import lfdpr, scenes as S
from parity import check_sampling, check_views, gpu_frame

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19901_gb300 import build
    build.build()
    lfdpr.lib()


def _mesh(triangles, texels=256):
    """Displaced surfaces of 5,000 triangles each, cut to the number asked for."""
    sc = S.geometry_paper(n_instances=-(-triangles // 5000), res=50, n_textures=2, seed=5, r_max=0.5)
    return replace(sc, idx=sc.idx[:triangles], tri_tex=sc.tri_tex[:triangles],
                   textures=[S.value_noise_texture(max(64, texels // 4), max(64, texels // 4), 7), S.value_noise_texture(texels, texels, 8)])


def _check(views, triangles, bias_h=1.0, bias_v=1.0, size=96, texels=256):
    d = replace(S.display_paper(), n_views=views, view_w=size, view_h=size + 8, focal_w=2.4 * size / (size + 8),
                bias_h=bias_h, bias_v=bias_v)
    sc, m = _mesh(triangles, texels), S.model_matrix(4)
    looked_at = sorted({0, views // 2, views - 1})
    o = O.render(d, sc, m, views=looked_at, panel=False)
    n = len(o.points)
    with lfdpr.Renderer(d, sc, n + 1) as R:
        g = gpu_frame(d, sc, m, renderer=R, panel=False)
        lfdpr.lfdpr_set_splat_lane_limit(R.disp, 3)
        walked = gpu_frame(d, sc, m, renderer=R, panel=False)
    assert g.stats.n_splat_writes > 0
    check_sampling(g, o)
    check_views(g, o, views=looked_at)
    assert walked.stats.n_splat_writes == g.stats.n_splat_writes
    assert np.array_equal(walked.keys, g.keys)
    return n


@pytest.mark.parametrize("views,triangles", [(49, 49999), (49, 50000), (64, 49999), (64, 50000), (65, 149999),
                                             (65, 150000), (96, 149999), (96, 150000)])
def test_meshes_on_either_side_of_a_line(views, triangles):
    _check(views, triangles)


@pytest.mark.parametrize("triangles,bias_h,bias_v", [(150000, 2.0, 1.0), (220000, 2.0, 1.0), (120000, 0.5, 1.0)])
def test_the_line_moves_with_the_bias(triangles, bias_h, bias_v):
    _check(70, triangles, bias_h, bias_v)


# views, triangles, bias: coarse cells with eight slots
@pytest.mark.parametrize("views,triangles,bias_h,bias_v", [(97, 20000, 4.0, 2.0), (128, 20000, 4.0, 4.0),
                                                           (130, 600, 8.0, 2.0)])
def test_coarse_cells_of_many_views(views, triangles, bias_h, bias_v):
    _check(views, triangles, bias_h, bias_v)


# views, triangles, bias, view size: up to 48 views, units by the points a warp has
@pytest.mark.parametrize("views,triangles,bias_h,bias_v,size", [(8, 10000, 4.0, 2.0, 160), (16, 20000, 8.0, 4.0, 200),
                                                                (8, 5000, 6.0, 1.0, 96), (4, 300, 1.0, 1.0, 64),
                                                                (24, 10000, 4.0, 2.0, 160), (48, 10000, 8.0, 4.0, 160),
                                                                (48, 50000, 4.0, 4.0, 96)])
def test_units_by_the_points(views, triangles, bias_h, bias_v, size):
    _check(views, triangles, bias_h, bias_v, size)


# views, view size: points on either side of the line between units of points
# from all over the list and of neighbours (1.2, 0.8 and 1.2 million points for one, two
# and three slots)
@pytest.mark.parametrize("views,size,least,most", [(48, 140, 3e5, 1.2e6), (40, 300, 2.4e6, 6e6), (24, 120, 3e5, 8e5),
                                                   (24, 300, 2.4e6, 6e6), (8, 140, 3e5, 1.2e6), (8, 300, 2.4e6, 6e6)])
def test_many_points(views, size, least, most):
    assert least < _check(views, 100000, 0.2, 0.2, size, 2048) < most
