"""The whole forward pass on views so wide that the layers keep no shared memory
free for the warp, and on the widest that do (12 input views: 720 pixels and
more do not), as tests/test_gpu_recon.py holds it to its reference."""
import pytest

from test_gpu_recon import test_forward_matches_reference as forward_matches_reference
from test_gpu_recon import torch  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,w", [(24, 712), (24, 720), (17, 901), (40, 1024)])
def test_wide_views(torch, h, w):  # noqa: F811
    forward_matches_reference(torch, h, w)
