"""The splat's units and blocks: view counts at the edges of every number of view
slots a lane, work lists from a few points to beyond a wave of blocks (where the
splat takes more blocks); sampling equals the oracle's and so do the views looked
at."""
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


# views, horizontal sampling bias (lower: more points)
@pytest.mark.parametrize("views,bias", [(1, 2.0), (16, 2.0), (17, 2.0), (32, 4.0), (33, 2.0), (48, 4.0), (49, 2.0),
                                        (64, 4.0), (65, 4.0), (96, 2.0), (97, 4.0), (128, 4.0), (16, 0.05),
                                        (33, 0.08), (96, 0.1), (8, 0.12), (24, 0.2), (48, 0.25), (60, 0.2)])
def test_views_equal_the_oracles(views, bias):
    d = replace(S.display_tiny(), n_views=views, view_w=96, view_h=96, bias_h=bias, bias_v=min(bias, 1.0))
    sc, m = S.scene_tiny(), S.model_matrix(4)
    looked_at = sorted({0, views // 2, views - 1})
    o = O.render(d, sc, m, views=looked_at, panel=False)
    g = gpu_frame(d, sc, m, max_points=len(o.points) + 1, panel=False)
    check_sampling(g, o)
    check_views(g, o, views=looked_at)


# views, bias, triangles: coarse cells (small units), and fewer points than warps
@pytest.mark.parametrize("views,bias,n", [(8, 12.0, 2048), (24, 12.0, 2048), (40, 30.0, 2048), (60, 12.0, 600),
                                          (90, 12.0, 2048), (120, 12.0, 300), (8, 2.0, 3), (40, 2.0, 50), (24, 60.0, 5)])
def test_few_points_and_coarse_cells(views, bias, n):
    d = replace(S.display_tiny(), n_views=views, view_w=160, view_h=160, bias_h=bias, bias_v=max(1.0, bias / 4))
    whole = S.scene_tiny()
    sc = replace(whole, idx=whole.idx[-n:], tri_tex=whole.tri_tex[-n:])
    m = S.model_matrix(4)
    looked_at = sorted({0, views // 2, views - 1})
    o = O.render(d, sc, m, views=looked_at, panel=False)
    g = gpu_frame(d, sc, m, max_points=len(o.points) + 1, panel=False)
    assert len(o.points) > 0
    check_sampling(g, o)
    check_views(g, o, views=looked_at)
