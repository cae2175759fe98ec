"""Batches of more scenes than branches, where a branch's next scene is sampled
while its last one is splatted: every scene's keys, views and panel equal the
frame alone, over consecutive frames and branch counts around the scenes'
number (a branch of two streams, and of one)."""
from dataclasses import replace

import numpy as np
import pytest

from paper_2601_19901_gb300 import lfdpr, scenes as S
from test_gpu_batch import _batched, _single

pytestmark = pytest.mark.gpu

N = 7


@pytest.fixture(scope="module")
def batch():
    import torch
    assert torch.cuda.is_available()
    from paper_2601_19901_gb300 import build
    build.build()
    ds = [replace(S.display_tiny(), n_views=(8, 40, 20, 70)[k % 4], view_w=64 + 8 * k, view_h=96, panel_w=256,
                  panel_h=128, recon=1 if k == 2 else 0, ss_level=1 if k == 3 else 0) for k in range(N)]
    scs = [S.scene_tiny(seed_mesh=k) for k in range(N)]
    for k in (1, 4):   # an empty mesh among them, and a very small one
        n = 0 if k == 1 else 3
        scs[k] = replace(scs[k], idx=scs[k].idx[:n], tri_tex=scs[k].tri_tex[:n])
    ts = lfdpr.TextureSet(scs[0].textures)
    B = lfdpr.Batch(ds, scs, ts, max_points=[1 << 18] * N)
    yield ds, scs, B
    B.close()
    ts.close()


@pytest.mark.parametrize("branches", [1, 2, 6, 7, 16, 2])
def test_scenes_equal_the_frames_alone(batch, branches):
    ds, scs, B = batch
    B.set_config(branches, 16, 6)
    for frame in (3, 11):
        models = np.stack([S.model_matrix(frame + 4 * k) for k in range(N)]).astype(np.float32)
        for _ in range(3):   # replays one after the other
            B.render(models)
        for i in range(N):
            got, ref = _batched(B, i, ds[i]), _single(ds[i], scs[i], models[i])
            assert got[0] == ref[0], i
            for a, b in zip(got[1:], ref[1:]):
                assert np.array_equal(a, b), i
    ms = B.scene_ms()
    assert np.all(ms > 0.0) and np.all(np.isfinite(ms))
