"""The shading frame of a point (its normal, tangent, the bitangent's sign, and the
normal map's values), which the materials' fetch stores for the resolve: texture
coordinates turned by any angle and mirrored in half of the triangles, strongly
tilted normal maps and a light along the surface, so that a wrong sign, axis or
map value moves colours by tens of levels; the views equal the oracle's."""
from dataclasses import replace

import numpy as np
import pytest

import oracle as O
from paper_2601_19901_gb300 import lfdpr, scenes as S
from parity import COLOUR_MAX_ABS, check_sampling, check_views, gpu_frame

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19901_gb300 import build
    build.build()
    lfdpr.lib()


def _scene(seed):
    rng = np.random.default_rng(seed)
    sc = S.scene_pbr_tiny()
    uv = sc.uv[sc.idx.ravel()].reshape(-1, 3, 2).astype(np.float64)
    n = len(uv)
    a, mirror = rng.uniform(0, 2 * np.pi, n), rng.random(n) < 0.5
    turn = np.stack([np.cos(a), -np.sin(a), np.sin(a), np.cos(a)], 1).reshape(n, 2, 2)
    turn[mirror, 0] *= -1.0
    uv = np.einsum("tij,tkj->tki", turn, uv)
    tex = []
    for k, t in enumerate(sc.textures):
        t = t.copy()
        if k % 4 == 1:      # normal maps: tilted by 30 to 60 degrees in every direction
            phi = rng.uniform(0, 2 * np.pi, t.shape[:2])
            tilt = rng.uniform(np.pi / 6, np.pi / 3, t.shape[:2])
            v = np.stack([np.sin(tilt) * np.cos(phi), np.sin(tilt) * np.sin(phi), np.cos(tilt)], -1)
            t[..., :3] = np.round((v * 0.5 + 0.5) * 255)
        tex.append(t)
    return replace(sc, xyz=sc.xyz[sc.idx.ravel()], uv=uv.reshape(-1, 2).astype(np.float32),
                   idx=np.arange(3 * n, dtype=np.uint32).reshape(-1, 3), textures=tex)


@pytest.mark.parametrize("seed", [0, 1])
def test_turned_and_mirrored_texture_coordinates(seed):
    sc = _scene(seed)
    d = replace(S.display_tiny(), bias_h=1.0)
    sh, m = S.Shading(light_dir=(0.8, 0.5, 0.3), light_rgb=(2.5, 2.5, 2.5), ambient=(0.02, 0.02, 0.02)), S.model_matrix(3)
    looked_at = [0, d.n_views // 2, d.n_views - 1]
    o = O.render(d, sc, m, views=looked_at, shading=sh, panel=False)
    with lfdpr.Renderer(d, sc, len(o.points) + 1, shading=sh) as R:
        g = gpu_frame(d, sc, m, renderer=R, panel=False)
    check_sampling(g, o)
    check_views(g, o, views=looked_at)
    # the oracle with the bitangent the other way (the maps' green inverted) differs
    wrong = [t.copy() for t in sc.textures]
    for k in range(1, len(wrong), 4):
        wrong[k][..., 1] = 255 - wrong[k][..., 1]
    w = O.render(d, replace(sc, textures=wrong), m, views=looked_at, shading=sh, panel=False)
    drawn = o.rgba[..., 3] > 0
    far = np.abs(o.rgba.astype(int) - w.rgba.astype(int)).max(-1) > 8 * COLOUR_MAX_ABS
    assert far[drawn].mean() > 0.5
