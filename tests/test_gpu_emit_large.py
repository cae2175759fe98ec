"""Meshes of few triangles, all of them large: shared out over the blocks that a
256-triangle block is spread to, among small ones emitted by their threads; the
point set equals the oracle's."""
import numpy as np
import pytest

from dataclasses import replace

import test_gpu_emit as emit
from test_gpu_emit import _lib  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,every,bias", [(1, 1, 0.5), (8, 1, 1.0), (9, 1, 0.5), (33, 1, 2.0), (200, 1, 4.0),
                                          (200, 7, 2.0), (256, 8, 2.0), (300, 31, 2.0)])
def test_the_point_set_is_the_oracles(n, every, bias, monkeypatch):
    def scene(count, seed, largest):
        rng = np.random.default_rng(seed)
        size = np.where(np.arange(n) % every == 0, largest, 0.02).reshape(n, 1, 1)
        tris = rng.uniform(-0.5, 0.5, (n, 1, 3)) + size * rng.uniform(-0.5, 0.5, (n, 3, 3))
        return replace(emit.S.scene_tiny(), xyz=tris.reshape(-1, 3).astype(np.float32),
                       uv=rng.uniform(0, 1, (3 * n, 2)).astype(np.float32),
                       idx=np.arange(3 * n, dtype=np.uint32).reshape(n, 3), tri_tex=np.zeros(n, np.uint32),
                       textures=[emit.S.value_noise_texture(64, 64, 7)])
    monkeypatch.setattr(emit, "_scene", scene)
    emit.test_the_point_set_is_the_oracles(n, bias, 1.4)
    emit.test_the_allocation_free_point_set_is_the_oracles(n, bias, 1.4)
