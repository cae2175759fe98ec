"""The interleave's forms against the oracle, byte for byte, on views of
random bytes.
"""
from dataclasses import replace

import numpy as np
import pytest

import oracle as O
from paper_2601_19901_gb300 import lfdpr, scenes as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_19901_gb300 import build
    build.build()
    lfdpr.lib()
    O.build()


def _display(n, w, h, pw, ph, pitch, slant, recon, xtalk):
    return replace(S.display_paper(), n_views=n, view_w=w, view_h=h, panel_w=pw, panel_h=ph, lens_pitch_px=pitch,
                   slant=slant, phase_offset=0.37, recon=recon, crosstalk=xtalk)


def _panel(d, views, jitter=None, samples=None):
    import torch
    disp = lfdpr.create_display(d, 16)
    mesh = None
    try:
        sc = S.scene_tiny()
        mesh = lfdpr.lfdpr_upload_mesh(disp, sc.xyz, sc.uv, sc.idx, sc.tri_tex, sc.textures)
        if jitter is not None:
            lfdpr.lfdpr_set_view_jitter(disp, jitter)
        if samples is not None:
            lfdpr.lfdpr_set_recon_samples(disp, samples)
        b = lfdpr.lfdpr_get_buffers(disp, mesh)
        lfdpr.device_view(b.views, views.shape, np.uint8).copy_(torch.from_numpy(views))
        panel = torch.full((d.panel_h, d.panel_w, 4), 7, dtype=torch.uint8, device="cuda")
        lfdpr.lfdpr_interleave(disp, panel.data_ptr(), torch.cuda.current_stream())
        torch.cuda.synchronize()
        return panel.cpu().numpy()
    finally:
        if mesh is not None:
            lfdpr.lfdpr_destroy_mesh(mesh)
        lfdpr.lfdpr_destroy_display(disp)


def _views(d, seed):
    return np.random.default_rng(seed).integers(0, 256, (d.n_render_views, d.view_h, d.view_w, 4), dtype=np.uint8)


@pytest.mark.parametrize("recon", [2, 3])
def test_sample_offsets_of_any_size(recon):
    """Angular offsets beyond every integer: all views are then equally near
    in binary32, as they are at 1e9, and the ends of the window answer."""
    d = _display(16, 12, 12, 260, 20, 8.0, 0.2, recon, 0.15)
    u = np.full(d.n_render_views, 0.5, np.float32)
    views = _views(d, recon)
    smp = np.zeros((4, 3), np.float32)
    smp[:, 2] = [0.0, 0.25, 1e30, -1e30]
    far = smp.copy()
    far[:, 2] = [0.0, 0.25, 1e9, -1e9]
    assert np.array_equal(_panel(d, views, u, smp), O.interleave(d, views, jitter=u, samples=far))
