"""Both kernels of the warp on either side of the rule between them (narrow rows
and few views a row, or not), against the restatement of test_gpu_warp, byte for
byte."""
import pytest

from test_gpu_warp_forms import _lib  # noqa: F401
from test_gpu_warp_forms import test_warp_forms_match_the_restatement as forms_match_the_restatement

pytestmark = pytest.mark.gpu


# (input views, output views, rows, columns)
@pytest.mark.parametrize("nin,nout,H,W", [(6, 30, 3, 110), (6, 30, 3, 111), (4, 60, 3, 192), (4, 60, 3, 193),
                                          (3, 60, 3, 224), (3, 60, 3, 225), (5, 18, 3, 256), (5, 17, 3, 256),
                                          (5, 20, 3, 128), (12, 60, 2, 223), (12, 49, 2, 225), (12, 21, 2, 400),
                                          (12, 22, 2, 400), (3, 40, 2, 401), (2, 1, 2, 333), (33, 60, 2, 512),
                                          (33, 60, 2, 513), (48, 2, 3, 180), (2, 300, 2, 33), (300, 40, 1, 20),
                                          (40, 320, 1, 130)])
def test_either_kernel(nin, nout, H, W):
    forms_match_the_restatement(nin, nout, H, W)
