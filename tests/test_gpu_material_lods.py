"""LOD pairs of a material's maps from one logarithm of the record's bounds:
texture coordinates from degenerate over tiny to huge (bounds of zero,
subnormal, ordinary and past the largest level's), maps of 1 to 256 texels a
side, square and not; the fetched values equal the oracle's exactly."""
from dataclasses import replace

import numpy as np
import pytest

import oracle as O
from paper_2601_19901_gb300 import lfdpr, scenes as S
from parity import check_sampling, gpu_frame
from test_gpu_pbr import _gpu_tvx, _oracle_tvx_r

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19901_gb300 import build
    build.build()
    lfdpr.lib()


@pytest.mark.parametrize("seed", range(3))
def test_fetched_values_equal_the_oracles(seed):
    rng = np.random.default_rng(seed)
    sc = S.scene_pbr_tiny()
    scale = rng.choice([0.0, 1e-22, 1e-19, 1e-12, 1e-3, 1.0, 50.0, 1e9], sc.n_tris)
    uv = sc.uv[sc.idx.ravel()].reshape(-1, 3, 2) * scale[:, None, None]
    sides = [(1, 1), (256, 1), (1, 128), (32, 64), (256, 256), (2, 16), (8, 8), (64, 4)]
    rng.shuffle(sides)
    sc = replace(sc, xyz=sc.xyz[sc.idx.ravel()], uv=uv.reshape(-1, 2).astype(np.float32),
                 idx=np.arange(3 * sc.n_tris, dtype=np.uint32).reshape(-1, 3),
                 textures=[rng.integers(0, 256, (h, w, 4)).astype(np.uint8) for w, h in sides])
    d, sh, m = S.display_tiny(), S.Shading(), S.model_matrix(2 + seed)
    o = O.render(d, sc, m, views=[0], shading=sh, panel=False)
    with lfdpr.Renderer(d, sc, len(o.points) + 1, shading=sh) as R:
        g = gpu_frame(d, sc, m, renderer=R, panel=False)
        tvx = _gpu_tvx(R, g.points.shape[0])
    check_sampling(g, o)
    assert np.array_equal(tvx, _oracle_tvx_r(o.tvx))
