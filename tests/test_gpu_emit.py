"""Point emission: triangles of one to hundreds of points, of one to dozens of
columns, in meshes at the edges of the rule that spreads a 256-triangle block
over several thread blocks; the point set equals the oracle's exactly. Both the
renderer (columns from the setup's summary) and the allocation-free entry point
(every triangle's columns walked)."""
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


def _scene(n, seed, largest):
    rng = np.random.default_rng(seed)
    size = 10.0 ** rng.uniform(-2.0, np.log10(largest), (n, 1, 1))
    size[: min(n, 3)] = largest                      # the first ones surely large
    tris = rng.uniform(-0.6, 0.6, (n, 1, 3)) + size * rng.uniform(-0.5, 0.5, (n, 3, 3))
    return S.Scene(xyz=tris.reshape(-1, 3).astype(np.float32),
                   uv=rng.uniform(0, 1, (3 * n, 2)).astype(np.float32),
                   idx=np.arange(3 * n, dtype=np.uint32).reshape(n, 3), tri_tex=np.zeros(n, np.uint32),
                   textures=[S.value_noise_texture(64, 64, 7)])


# triangles, horizontal sampling bias, largest triangle
CASES = [(1, 0.5, 1.5), (2, 4.0, 1.5), (255, 0.5, 1.2), (256, 1.0, 1.2), (257, 4.0, 1.2), (38 * 256, 1.0, 0.3),
         (38 * 256 + 1, 2.0, 0.3), (76 * 256 + 3, 2.0, 0.2), (152 * 256 + 1, 1.0, 0.7), (153 * 256 + 7, 4.0, 0.3)]


@pytest.mark.parametrize("n,bias,largest", CASES)
def test_the_point_set_is_the_oracles(n, bias, largest):
    import torch
    d = replace(S.display_tiny(), bias_h=bias)
    sc = _scene(n, n, largest)
    m = S.model_matrix(2)
    _, tri, want_counts = O.setup(d, sc, m)
    want = O.emit(tri, want_counts)
    total = int(want_counts.sum())
    s = torch.cuda.current_stream()
    with lfdpr.Renderer(d, sc, total + 5) as R:
        R.render(m, s)
        st = R.stats(s)
        assert st.n_points == total and not st.overflow
        b = R.buffers()
        assert np.array_equal(lfdpr.device_to_numpy(b.counts, (n,), np.uint32), want_counts)
        got = lfdpr.device_to_numpy(b.points, (total, 4), np.uint32) if total else np.zeros((0, 4), np.uint32)
        assert np.array_equal(got[:, :2], want[:, :2])


@pytest.mark.parametrize("n,bias,largest", CASES[:7])
def test_the_allocation_free_point_set_is_the_oracles(n, bias, largest):
    import torch
    d = replace(S.display_tiny(), bias_h=bias)
    sc = _scene(n, 7 * n, largest)
    m = S.model_matrix(2)
    _, tri, want_counts = O.setup(d, sc, m)
    want = O.emit(tri, want_counts)
    total = int(want_counts.sum())
    s = torch.cuda.current_stream()
    dev = torch.device("cuda")
    xyz, uv = torch.from_numpy(sc.xyz).to(dev), torch.from_numpy(sc.uv).to(dev)
    idx, tex = torch.from_numpy(sc.idx.astype(np.int32)).to(dev), torch.from_numpy(sc.tri_tex.astype(np.int32)).to(dev)
    pts = torch.zeros((total + 5, 4), dtype=torch.int32, device=dev)
    counts = torch.zeros(n, dtype=torch.int32, device=dev)
    fc = torch.zeros(4, dtype=torch.int32, device=dev)
    lfdpr.lfdpr_sample_points_noalloc(lfdpr.desc_of(d), m, xyz.data_ptr(), uv.data_ptr(), idx.data_ptr(),
                                      tex.data_ptr(), n, np.array([[64, 64]], np.uint32), pts.data_ptr(), total + 5,
                                      counts.data_ptr(), fc.data_ptr(), s)
    torch.cuda.synchronize()
    assert int(fc[0]) == total and int(fc[1]) == 0
    assert np.array_equal(counts.cpu().numpy().view(np.uint32), want_counts)
    got = pts.cpu().numpy().view(np.uint32)
    assert np.array_equal(got[:total, :2], want[:, :2]) and not got[total:].any()


# blocks of triangles where a block's sums over the blocks before it end (2,048), and one past
@pytest.mark.parametrize("blocks,over", [(2048, 0), (2048, 1), (1, 0), (5, 7)])
@pytest.mark.parametrize("short", [0, 1])
def test_counters_and_offsets_of_whole_meshes(blocks, over, short):
    import torch
    n = 256 * blocks + over
    d = replace(S.display_tiny(), bias_h=4.0, bias_v=4.0)
    rng = np.random.default_rng(n)
    tris = rng.uniform(-0.9, 0.9, (n, 1, 3)) + 0.02 * rng.uniform(-1, 1, (n, 3, 3))
    tris[rng.random(n) < 0.1] += 40.0                 # some out of sight
    sc = S.Scene(xyz=tris.reshape(-1, 3).astype(np.float32), uv=rng.uniform(0, 1, (3 * n, 2)).astype(np.float32),
                 idx=np.arange(3 * n, dtype=np.uint32).reshape(n, 3), tri_tex=np.zeros(n, np.uint32),
                 textures=[S.value_noise_texture(64, 64, 7)])
    m = np.eye(4, dtype=np.float32)
    _, tri, want = O.setup(d, sc, m)
    total, live = int(want.sum()), int((tri[:, O.F["live"]] == 1).sum())
    offsets = np.concatenate([[0], np.cumsum(want.astype(np.int64))[:-1]])
    assert 0 < live < n or n < 300
    s = torch.cuda.current_stream()
    with lfdpr.Renderer(d, sc, total - short) as R:
        for _ in range(2):                            # the second frame finds the first one's counters
            R.render(m, s)
            if short:
                with pytest.raises(lfdpr.LfdprError, match="needed %d points" % total):
                    R.stats(s)
            else:
                st = R.stats(s)
                assert (st.n_points, st.n_live_tris, st.overflow, st.cell_overflow) == (total, live, 0, 0)
            b = R.buffers()
            assert np.array_equal(lfdpr.device_to_numpy(b.offsets, (n,), np.uint32), offsets)
            if not short:
                got = lfdpr.device_to_numpy(b.points, (total, 4), np.uint32)
                assert np.array_equal(got[:, :2], O.emit(tri, want)[:, :2])
