"""Mip levels of the rendered views (spatial supersampling): rows shorter than a
warp's stretch, ending inside one and filling some exactly, few rows and many,
both levels; the panel equals the oracle's interleave of the same views."""
from dataclasses import replace

import numpy as np
import pytest

import oracle as O
from paper_2601_19901_gb300 import lfdpr, scenes as S
from parity import gpu_frame

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19901_gb300 import build
    build.build()
    lfdpr.lib()


@pytest.mark.parametrize("level,w,h,views,recon", [(1, 2, 2, 1, 0), (1, 62, 10, 3, 0), (1, 64, 64, 8, 0), (1, 126, 34, 5, 1),
                                                   (1, 130, 66, 5, 0), (1, 258, 130, 48, 0), (2, 4, 4, 1, 0),
                                                   (2, 60, 12, 3, 0), (2, 128, 132, 4, 1), (2, 132, 128, 9, 0),
                                                   (2, 516, 260, 48, 0)])
def test_the_panel_of_view_mips_is_the_oracles(level, w, h, views, recon):
    d = replace(S.display_tiny(), n_views=views, view_w=w, view_h=h, ss_level=level, recon=recon, bias_h=1.0)
    g = gpu_frame(d, S.scene_tiny(), S.model_matrix(3), max_points=1 << 20)
    assert not g.stats.overflow and g.stats.n_points > 0
    assert np.array_equal(g.panel, O.interleave(d, g.views))
