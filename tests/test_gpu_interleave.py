"""The interleave's forms against the oracle, byte for byte, on views of
random bytes: sizes at which a strip of panel columns, a lens period or a
view row is left over, one view and many, eyes placed on the same border of
their intervals (no threshold separates them) and sample offsets beyond the
table of nearest views.
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


# (views, view w, h, panel w, h, pitch, slant, recon, crosstalk, samples, eyes, largest dphi)
GAUSS = [(48, 42, 56, 256, 16, 8.0, 0.2, 2, 0.15, 8, "random", None),      # one whole strip
         (48, 42, 56, 257, 17, 8.0, 0.2, 2, 0.15, 8, "random", None),      # and one column more
         (48, 21, 28, 1600, 9, 8.0, -0.2, 3, 0.15, 8, "random", None),
         (37, 33, 25, 1277, 13, 5.3, 1.0 / 6.0, 2, 0.0, 7, "random", None),
         (24, 64, 20, 900, 11, 5.0, 0.25, 2, 0.15, 32, "half", None),
         (8, 17, 9, 31, 300, 2.5, 0.1, 3, 0.1, 1, "random", None),
         (1, 9, 9, 40, 10, 8.0, 0.2, 3, 0.2, 3, "random", None),
         (1, 9, 9, 40, 10, 8.0, 0.2, 2, 0.2, 4, "random", None),
         (2, 5, 3, 70, 10, 4.0, 0.0, 2, 0.3, 8, "random", None),
         (256, 8, 8, 520, 8, 11.0, 0.3, 2, 0.15, 8, "random", None),       # the most views
         (16, 12, 12, 260, 20, 8.0, 0.2, 2, 0.15, 8, "ends", None),        # every interval's start or end
         (16, 12, 12, 260, 20, 8.0, 0.2, 2, 0.15, 8, "border", None),      # neighbours at one place
         (16, 12, 12, 260, 20, 8.0, 0.2, 3, 0.15, 8, "border", None),
         (16, 12, 12, 260, 20, 8.0, 0.2, 2, 0.15, 8, "close", None),       # neighbours a few floats apart
         (16, 12, 12, 260, 20, 8.0, 0.2, 2, 0.15, 8, "random", 4.0),       # the table's last bin
         (16, 12, 12, 260, 20, 8.0, 0.2, 2, 0.15, 8, "random", 4.01),      # beyond it
         (16, 12, 12, 260, 20, 8.0, 0.2, 2, 0.15, 8, "random", 1e9)]


@pytest.mark.parametrize("case", range(len(GAUSS)))
def test_gaussian_interleave_matches_oracle(case):
    n, w, h, pw, ph, pitch, slant, recon, xtalk, ns, eyes, dphi = GAUSS[case]
    d = _display(n, w, h, pw, ph, pitch, slant, recon, xtalk)
    rng = np.random.default_rng(100 + case)
    nr = d.n_render_views
    u = {"random": rng.random(nr), "half": np.full(nr, 0.5), "ends": rng.integers(0, 2, nr).astype(float),
         "border": np.arange(nr) % 2 == 0, "close": np.where(np.arange(nr) % 2 == 0, 1.0 - 1e-6, 1e-6)}[eyes]
    u = np.asarray(u).astype(np.float32)
    smp = (rng.normal(0.0, 1.0, (ns, 3)) * [0.5625, 0.5625, 0.5]).astype(np.float32)
    if dphi is not None:
        smp[0, 2], smp[1, 2] = dphi, -dphi
    views = _views(d, case)
    assert np.array_equal(_panel(d, views, u, smp), O.interleave(d, views, jitter=u, samples=smp))


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


# (views, view w, h, panel w, h, pitch, slant, recon, crosstalk)
TILED = [(48, 42, 56, 512, 33, 8.0, 0.2, 1, 0.15),        # one whole strip of panel columns
         (48, 42, 56, 513, 33, 8.0, 0.2, 1, 0.15),        # two, uneven
         (48, 42, 56, 2560, 12, 8.0, 0.2, 1, 0.0),
         (37, 33, 25, 1277, 13, 5.3, 1.0 / 6.0, 1, 0.2),
         (37, 33, 25, 1277, 13, 5.3, 1.0 / 6.0, 0, 0.2),
         (37, 33, 25, 1278, 130, 5.3, -0.3, 0, 0.0),
         (3, 40, 30, 77, 20, 2.5, 0.1, 1, 0.4),
         (2, 40, 30, 77, 20, 2.5, 0.1, 1, 0.4),
         (1, 40, 30, 77, 20, 2.5, 0.1, 1, 0.4),
         (1, 1, 1, 1, 1, 1.0, 0.0, 1, 0.1),
         (5, 300, 200, 30, 20, 6.0, 0.1, 1, 0.1),         # more view pixels than panel pixels
         (40, 2000, 4, 100, 40, 8.0, 0.2, 1, 0.15),       # no tile fits: the direct gather
         (256, 12, 9, 260, 20, 9.0, 0.2, 1, 0.15)]


@pytest.mark.parametrize("case", range(len(TILED)))
def test_tiled_interleave_matches_oracle(case):
    d = _display(*TILED[case])
    views = _views(d, 50 + case)
    assert np.array_equal(_panel(d, views), O.interleave(d, views))
