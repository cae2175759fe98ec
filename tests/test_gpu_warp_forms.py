"""The warp at the sizes where its sweeps and passes end: rows of one pixel,
of a block's threads and one more, several sweeps, more output views in one
interval than a pass takes, intervals without any, against the restatement
of test_gpu_warp, byte for byte."""
import numpy as np
import pytest

from test_gpu_warp import F32, NO_KEY, run_gpu, warp_reference

pytestmark = pytest.mark.gpu

# (input views, output views, rows, columns)
FORMS = [(2, 1, 1, 1), (2, 9, 3, 1), (2, 13, 5, 8), (5, 3, 4, 32), (12, 48, 3, 224), (12, 48, 3, 256), (3, 40, 4, 257),
         (4, 64, 3, 513), (2, 5, 2, 1500), (2, 130, 2, 2100), (40, 2, 2, 60)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19901_gb300 import build, lfdpr
    build.build()
    lfdpr.lib()


@pytest.mark.parametrize("nin,nout,H,W", FORMS)
def test_warp_forms_match_the_restatement(nin, nout, H, W):
    rng = np.random.default_rng(nin * 1000 + nout * 10 + W)
    in_eyes = np.sort(rng.uniform(-1.0, 1.0, nin)).astype(F32)
    out_eyes = rng.uniform(-1.1, 1.1, nout).astype(F32)
    t = rng.uniform(0.3, 3.0, (nin, H, W)).astype(F32)
    t[:, :, ::3] = F32(0.75)     # equal depths: the first input, then the leftmost pixel
    keys = (t.view(np.uint32).astype(np.uint64) << np.uint64(32)) | rng.integers(0, 1 << 20, (nin, H, W)).astype(np.uint64)
    keys[rng.random((nin, H, W)) < 0.2] = NO_KEY
    views = rng.integers(0, 256, (nin, H, W, 4), dtype=np.uint8)
    ipw = F32(rng.uniform(5.0, 60.0))
    got = run_gpu(views, keys, in_eyes, out_eyes, ipw)
    ref = warp_reference(views, keys, in_eyes, out_eyes, ipw)
    assert np.array_equal(got, ref), "bytes differ at %d pixels" % int((got != ref).any(-1).sum())
