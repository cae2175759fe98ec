"""The library's own choice of view bands: more than 64 views whose keys are far
beyond L2 are cleared, splatted and resolved in equal bands, with the keys and
views of one band; fewer views, or smaller ones, in one band (seen by the
frame's launches)."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2601_19901_gb300 import lfdpr, scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19901_gb300 import build
    build.build()
    lfdpr.lib()


# views, width, height, bands the library takes
@pytest.mark.parametrize("views,w,h,bands", [(65, 830, 830, 2), (72, 790, 800, 2), (72, 779, 780, 1), (64, 850, 850, 1),
                                             (129, 590, 600, 3)])
def test_the_librarys_bands_give_the_frame_of_one(views, w, h, bands):
    import torch
    d = replace(S.display_tiny(), n_views=views, view_w=w, view_h=h, bias_h=1.0)
    with lfdpr.Renderer(d, S.scene_tiny(), max_points=1 << 21) as R:
        s = torch.cuda.current_stream()

        def frame(band):
            lfdpr.lfdpr_set_view_band(R.disp, band)
            before = R.stats(s).kernel_launches
            R.render(S.model_matrix(7), s)
            st = R.stats(s)
            b = R.buffers()
            shape = (views, h, w)
            return (st.kernel_launches - before, st.n_points,
                    lfdpr.device_view(b.keys, shape, np.uint64).clone(),
                    lfdpr.device_view(b.views, shape + (4,), np.uint8).clone())

        n1, p1, k1, v1 = frame(views)
        n0, p0, k0, v0 = frame(0)
        assert p0 == p1 > 0
        assert n0 - n1 == 2 * (bands - 1)
        assert torch.equal(k0, k1) and torch.equal(v0, v1)
