"""The interleave's forms on either side of the rules that choose between them,
byte for byte against the oracle on views of random bytes: the tent's tiles
(panels of many rows a view row) and the gather, with and without crosstalk;
the Gaussian with and without its table; the plain tiles staged run after run
and view after view.
"""
import numpy as np
import pytest

import oracle as O
from test_gpu_interleave import _display, _lib, _panel, _views  # noqa: F401

pytestmark = pytest.mark.gpu

# (views, view w, h, panel w, h, pitch, slant, recon, crosstalk)
TENT = [(48, 42, 9, 512, 33, 8.0, 0.2, 1, 0.15),          # tiles: one whole strip of panel columns
        (48, 42, 9, 513, 34, 8.0, 0.2, 1, 0.15),          # two, uneven
        (37, 33, 25, 1277, 131, 5.3, 1.0 / 6.0, 1, 0.2),
        (24, 33, 80, 1277, 200, 5.3, 1.0 / 6.0, 1, 0.0),
        (8, 16, 90, 514, 270, 8.0, -0.2, 1, 0.0),
        (1, 40, 90, 515, 200, 2.5, 0.1, 1, 0.4),          # one view, whose neighbours are itself
        (1, 40, 90, 515, 200, 2.5, 0.1, 1, 0.0),
        (2, 40, 90, 515, 200, 2.5, 0.1, 1, 0.4),
        (3, 40, 90, 515, 200, 2.5, 0.1, 1, 0.4),
        (256, 12, 9, 260, 200, 9.0, 0.2, 1, 0.15),        # the most views
        (100, 240, 8, 1000, 80, 8.0, 0.2, 1, 0.15),       # more than 48 KB of shared memory
        (4, 12, 200, 1030, 100, 8.0, 0.2, 1, 0.15),       # tiles of one panel row
        (4, 12, 200, 1030, 100, 8.0, 0.2, 1, 0.0),
        (48, 42, 56, 512, 56, 8.0, 0.2, 1, 0.15),         # gather: a panel row per view row
        (96, 42, 56, 512, 120, 8.0, 0.2, 1, 0.0),         # gather: many views a panel pixel
        (200, 42, 20, 256, 60, 8.0, 0.2, 1, 0.15)]


@pytest.mark.parametrize("case", range(len(TENT)))
def test_tent_matches_oracle(case):
    d = _display(*TENT[case])
    views = _views(d, 80 + case)
    assert np.array_equal(_panel(d, views), O.interleave(d, views))


TILE = [(15, 129, 7, 1024, 9, 8.0, 0.2, 0, 0.0),      # view after view: the first segment longer than a run
        (15, 128, 7, 1024, 9, 8.0, 0.2, 0, 0.0),      # run after run
        (16, 129, 7, 1024, 9, 8.0, 0.2, 0, 0.0),
        (15, 300, 7, 1100, 9, 8.0, 0.2, 0, 0.3),      # a last strip of few columns
        (2, 1000, 5, 400, 3, 2.5, -0.1, 0, 0.0),      # views wider than the panel
        (1, 1000, 5, 1000, 5, 2.5, 0.1, 0, 0.4)]


@pytest.mark.parametrize("case", range(len(TILE)))
def test_tiles_match_oracle(case):
    d = _display(*TILE[case])
    views = _views(d, 160 + case)
    assert np.array_equal(_panel(d, views), O.interleave(d, views))


# (views, view w, h, panel w, h, pitch, slant, recon, crosstalk, samples, largest dphi)
GAUSS = [(48, 21, 28, 64, 64, 8.0, 0.2, 2, 0.0, 1, None),         # too little for a table
         (96, 21, 28, 65, 63, 8.0, 0.2, 3, 0.0, 2, None),
         (256, 8, 9, 130, 20, 11.0, 0.3, 2, 0.15, 2, None),
         (256, 8, 9, 130, 20, 11.0, 0.3, 2, 0.15, 3, None),       # enough for one
         (1, 9, 9, 1, 1, 8.0, 0.2, 2, 0.2, 1, None),
         (16, 12, 12, 700, 300, 8.0, 0.2, 2, 0.15, 7, 4.01),      # beyond the table
         (16, 12, 12, 700, 300, 8.0, 0.2, 3, 0.0, 8, -9.0)]


@pytest.mark.parametrize("case", range(len(GAUSS)))
def test_gaussian_matches_oracle(case):
    *size, ns, dphi = GAUSS[case]
    d = _display(*size)
    rng = np.random.default_rng(200 + case)
    u = rng.random(d.n_render_views).astype(np.float32)
    smp = (rng.normal(0.0, 1.0, (ns, 3)) * [0.5625, 0.5625, 0.5]).astype(np.float32)
    if dphi is not None:
        smp[-1, 2] = dphi
    views = _views(d, 120 + case)
    assert np.array_equal(_panel(d, views, u, smp), O.interleave(d, views, jitter=u, samples=smp))
