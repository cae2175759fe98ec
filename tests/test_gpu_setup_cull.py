"""Visibility of triangles about the side planes of the views' frusta: inside by
a hair, outside of one view, of some or of all, with displays of one to many
views; counts and records equal the oracle's exactly."""
from dataclasses import replace

import numpy as np
import pytest

import oracle as O
from paper_2601_19901_gb300 import lfdpr, scenes as S
from parity import check_sampling, gpu_frame

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19901_gb300 import build
    build.build()
    lfdpr.lib()


def _scene(d, n, seed):
    """Small triangles, each with one vertex on a side plane of a random view (an
    extreme one for half of them), moved off it by nothing, by a few last places
    or by up to a triangle's size to either side."""
    rng = np.random.default_rng(seed)
    eyes = np.asarray(O.eyes(d), np.float64)
    v = rng.integers(0, len(eyes), n)
    ends = rng.random(n) < 0.5
    v[ends] = np.where(rng.random(int(ends.sum())) < 0.5, 0, len(eyes) - 1)
    side = np.where(rng.random(n) < 0.5, -1.0, 1.0)
    z = rng.uniform(-3.0, 1.5, n)
    # the plane through the eye (e, 0, D) and the focal rectangle's side edge (side fw / 2, ., 0)
    x = eyes[v] + (side * 0.5 * d.focal_w - eyes[v]) * (d.view_dist - z) / d.view_dist
    off = rng.choice([0.0, 1e-7, -1e-7, 1e-6, -1e-6, 1e-2, -1e-2, 0.1, -0.1], n)
    y = rng.uniform(-0.6, 0.6, n)
    tri = np.zeros((n, 3, 3))
    tri[:, 0] = np.stack([x + off, y, z], 1)
    for k in (1, 2):   # the other vertices further out, or further in for a few
        tri[:, k] = tri[:, 0] + np.stack([side * rng.uniform(0, 0.1, n) * np.where(rng.random(n) < 0.9, 1, -1),
                                          rng.uniform(-0.1, 0.1, n), rng.uniform(-0.05, 0.05, n)], 1)
    return S.Scene(xyz=tri.reshape(-1, 3).astype(np.float32), uv=rng.uniform(0, 1, (3 * n, 2)).astype(np.float32),
                   idx=np.arange(3 * n, dtype=np.uint32).reshape(n, 3), tri_tex=np.zeros(n, np.uint32),
                   textures=[S.value_noise_texture(32, 32, 3)])


@pytest.mark.parametrize("views,cone,recon", [(1, 30.0, 0), (2, 40.0, 0), (7, 60.0, 0), (24, 40.0, 1), (48, 90.0, 1),
                                              (96, 40.0, 0)])
def test_triangles_about_the_side_planes(views, cone, recon):
    d = replace(S.display_tiny(), n_views=views, cone_deg=cone, recon=recon, view_w=64, view_h=64)
    sc = _scene(d, 3000, 10 * views + recon)
    m = np.eye(4, dtype=np.float32)
    o = O.render(d, sc, m, views=[0], panel=False)
    live = int((o.tri[:, O.F["live"]] == 1).sum())
    assert 300 < live < 2900     # both outcomes, many times
    check_sampling(gpu_frame(d, sc, m, panel=False), o)
