"""Performance cases: the frames a user of the library renders, each through
the public binding (paper_2601_19901_gb300.lfdpr), over the range of sizes,
view counts and options the library is used with.

A case is a dict of plain values. Its "kind" says what one pass is:

  frame    lfdpr_render_frame + lfdpr_interleave of one mesh on one display
           (plain, tent or Gaussian reconstruction, spatial supersampling,
           materials with physically based shading, device or host panel)
  batch    lfdpr_render_batch of several scenes, each on its own display
  learned  a quarter of the views rendered, lfdpr_recon_run, interleave
  network  lfdpr_recon_run alone, on views rendered beforehand
  sample   lfdpr_sample_points_noalloc, the point generation of a render loop
           that may not allocate

Every output is a whole number (8-bit colours, depth keys, point ids and
counts) that the library specifies down to the rounding of each binary32
operation, so there is no 64-bit value to compare them with: exact() has none,
and outputs are to be equal.
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

from paper_2601_19901_gb300 import lfdpr, recon_net, scenes as S

SIGMA = np.array([2.25 / 4, 2.25 / 4, 0.5])   # Gaussian sample offsets: dx, dy (pixels), dphi (views)


def _frame(name, **kw):
    """A frame case: by default the 48-view display and scene of the paper-shaped workload."""
    c = dict(name=name, kind="frame", instances=200, res=50, views=48, w=420, h=560, panel_w=2560, panel_h=1600,
             pitch=8.0, slant=0.2, recon=0, xtalk=0.0, ss=0, bias=1.0, textures=64, max_tex=4096, pbr=False,
             host=False)
    c.update(kw)
    return c


def listed():
    return [
        # the 2,048-triangle mesh on the 8-view display: the smallest frame, all launches and latency
        dict(name="tiny_frame", kind="frame", tiny=True, views=8, w=128, h=128, panel_w=512, panel_h=512, recon=0,
             ss=0),
        # point generation of a small mesh inside a render loop that may not allocate
        dict(name="sample_points", kind="sample", instances=8, res=45, views=48, w=420, h=560, textures=16),
        # a modest model on a display of odd sizes: 37 views of 333x251, a panel that no tile divides
        _frame("ragged_frame", instances=22, res=50, views=37, w=333, h=251, panel_w=1277, panel_h=719, pitch=5.3,
               slant=1.0 / 6.0, bias=1.5, textures=13, max_tex=1024),
        # a 300,000-triangle model, 48 views of 480x360, shown through pinned host memory (end to end)
        _frame("host_frame", instances=60, res=50, w=480, h=360, panel_w=1920, panel_h=1080, textures=24,
               max_tex=2048, host=True),
        # the paper-shaped frame: 10^6 triangles, 48 views of 420x560, 2560x1600 panel
        _frame("paper_frame"),
        # the same at twice the angular rate (96 views), tent reconstruction, crosstalk
        _frame("angular_frame", recon=1, xtalk=0.15),
        # the same at random angles, Gaussian reconstruction with 8 samples, crosstalk
        _frame("gauss_frame", recon=2, xtalk=0.15),
        # ... with 2x spatial supersampling as well: views of 840x1120
        _frame("gauss_spatial_frame", recon=2, xtalk=0.15, ss=1, w=840, h=1120),
        # materials of four textures, physically based shading
        _frame("pbr_frame", pbr=True),
        # twelve scenes of 5,000 to 200,000 triangles in one graph, displays of 24, 48 and 96 views
        dict(name="batch", kind="batch", scenes=12, tris_lo=5000, tris_hi=200000, textures=24, max_tex=1024),
        # the learned path: 12 of 48 views rendered, the rest predicted, interleaved
        _frame("learned_frame", kind="learned", xtalk=0.15),
        # its network alone, at a size that no tile divides
        _frame("network_ragged", kind="network", instances=40, w=333, h=251, textures=13, max_tex=1024),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["plain", "tent", "gauss", "spatial", "pbr", "host", "batch", "learned", "network", "sample"],
                       [3, 1, 1, 1, 1, 1, 1, 1, 1, 1])[0]
    if kind == "batch":
        lo = _log(rng, 2000, 20000)
        return dict(kind="batch", scenes=_log(rng, 3, 12), tris_lo=lo, tris_hi=lo * rng.randint(2, 8),
                    textures=rng.randint(4, 24), max_tex=1024)
    if kind == "sample":
        return dict(kind="sample", instances=rng.randint(2, 8), res=_log(rng, 8, 45), views=_log(rng, 5, 96),
                    w=_log(rng, 120, 640), h=_log(rng, 120, 640), textures=rng.randint(1, 64))
    tris = _log(rng, 2000, 1000000)
    inst = max(2, min(200, tris // 2000))
    c = _frame("", instances=inst, res=max(4, int(round(math.sqrt(tris / (2.0 * inst))))), views=_log(rng, 5, 96),
               w=_log(rng, 120, 640), h=_log(rng, 120, 640), panel_w=_log(rng, 400, 2560),
               panel_h=_log(rng, 300, 1600), pitch=round(rng.uniform(4.0, 10.0), 2),
               slant=round(rng.uniform(-0.25, 0.35), 3), bias=rng.choice([1.0, 1.0, 1.5, 2.0]),
               textures=rng.randint(1, 32), max_tex=2 ** rng.randint(8, 11))
    del c["name"]
    if kind in ("tent", "gauss", "spatial"):
        c.update(views=_log(rng, 5, 48), recon=1 if kind == "tent" else rng.choice([2, 2, 3]),
                 xtalk=rng.choice([0.0, 0.15]))
    if kind == "spatial":
        c.update(ss=1, w=2 * _log(rng, 100, 420), h=2 * _log(rng, 100, 560), recon=rng.choice([0, 1, 2]))
    if kind == "pbr":
        c.update(pbr=True)
    if kind == "host":
        c.update(host=True)
    if kind in ("learned", "network"):
        c.update(kind=kind, views=48, bias=1.0, xtalk=rng.choice([0.0, 0.15]))
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _noise(size, gen, channels=3, base=8, octaves=4):
    """Value noise in [0, 1], [channels][size][size] (float32, GPU): octaves of random periodic lattices."""
    acc = torch.zeros((channels, size, size), device="cuda")
    for k in range(octaves):
        n = min(base << k, size)
        g = torch.rand((1, channels, n, n), generator=gen, device="cuda")
        g = torch.cat([g, g[..., :1]], -1)
        g = torch.cat([g, g[..., :1, :]], -2)
        g = torch.nn.functional.interpolate(g, size=(size + 1, size + 1), mode="bilinear", align_corners=True)
        acc += 0.5 ** k * g[0, :, :size, :size]
    lo, hi = torch.aminmax(acc)
    return (acc - lo) / (hi - lo)


def _rgba(rgb):
    """RGBA8 [h][w][4] (numpy) of rgb [3][h][w] in [0, 1]."""
    out = torch.full(rgb.shape[1:] + (4,), 255, dtype=torch.uint8, device="cuda")
    out[..., :3] = (rgb * 255.0).round().clamp(0, 255).to(torch.uint8).permute(1, 2, 0)
    return out.cpu().numpy()


def _sizes(max_tex):
    return [1 << k for k in range(6, int(math.log2(max_tex)) + 1)]


def _textures(n, max_tex, seed):
    """n value-noise textures from 64^2 to max_tex^2 (powers of two, cycled)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    sizes = _sizes(max_tex)
    return [_rgba(_noise(sizes[k % len(sizes)], gen)) for k in range(n)]


def _materials(n, max_tex, seed):
    """n materials of four textures of different sizes: albedo, tangent-space
    normal map of a noise height field, roughness, a mostly binary metallic mask."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    sizes = _sizes(max_tex)
    out = []
    for m in range(n):
        sa, sn, sr, sm = (sizes[(m + 3 * j) % len(sizes)] for j in range(4))
        out.append(_rgba(_noise(sa, gen)))
        hgt = _noise(sn, gen, 1)[0]
        dx, dy = (4.0 * (torch.roll(hgt, -1, d) - torch.roll(hgt, 1, d)) for d in (1, 0))
        nrm = torch.stack([-2.0 * dx, -2.0 * dy, torch.ones_like(hgt)])
        out.append(_rgba(nrm / nrm.norm(dim=0, keepdim=True) * 0.5 + 0.5))
        out.append(_rgba((0.15 + 0.8 * _noise(sr, gen, 1)).expand(3, sr, sr)))
        out.append(_rgba(((_noise(sm, gen, 1) - 0.5) * 4.0 + 0.5).clamp(0, 1).expand(3, sm, sm)))
    return out


def _geometry(instances, res, n_tex, seed):
    """Displaced meshes with log-uniform radii; fewer instances are larger, so that they fill the views as well."""
    return S.geometry_paper(n_instances=instances, res=res, n_textures=n_tex, seed=seed,
                            r_max=min(0.7, 0.2 * math.sqrt(200.0 / instances)))


def _display(c, **kw):
    d = replace(S.display_paper(), n_views=c["views"], view_w=c["w"], view_h=c["h"], focal_w=2.4 * c["w"] / c["h"])
    if "panel_w" in c:
        d = replace(d, panel_w=c["panel_w"], panel_h=c["panel_h"], lens_pitch_px=c["pitch"], slant=c["slant"],
                    recon=c["recon"], crosstalk=c["xtalk"], ss_level=c["ss"], bias_h=c["bias"])
    return replace(d, **kw)


def _scene(c, seed):
    if c.get("tiny"):
        return S.scene_tiny(seed_mesh=seed, seed_tex=seed + 1)
    if c["pbr"]:
        n = max(1, c["textures"] // 4)
        sc = _geometry(c["instances"], c["res"], n, seed)
        sc.textures = _materials(n, c["max_tex"], seed)
        sc.materials = np.arange(4 * n, dtype=np.uint32).reshape(n, 4)
        return sc
    sc = _geometry(c["instances"], c["res"], c["textures"], seed)
    sc.textures = _textures(c["textures"], c["max_tex"], seed)
    return sc


class _Held:
    """The library's objects of a state, closed in order when the last tensor over their memory goes."""

    def __init__(self, *objects):
        self.objects = objects

    def __del__(self):
        for o in self.objects:
            o.close()


class _Display:
    """A display without a mesh (the target of the learned path)."""

    def __init__(self, d):
        self.disp = lfdpr.create_display(d, 1)

    def close(self):
        lfdpr.lfdpr_destroy_display(self.disp)


class _Memory:
    """Device memory of a held object, for torch: the tensor keeps the object."""

    def __init__(self, held, ptr, shape, typestr):
        self.held = held
        self.__cuda_array_interface__ = dict(shape=shape, typestr=typestr, data=(ptr, False), version=3, strides=None)


def _of_display(held, disp, nr, d, with_keys=True):
    """The views and depth keys of display `disp`, as tensors over its own buffers."""
    out = {"views": torch.as_tensor(_Memory(held, disp.views, (nr, d.view_h, d.view_w, 4), "|u1"), device="cuda")}
    if with_keys:
        out["keys"] = torch.as_tensor(_Memory(held, disp.keys, (nr, d.view_h, d.view_w), "<i8"), device="cuda")
    return out


def _buffers(disp, mesh):
    return lfdpr.lfdpr_get_buffers(disp, mesh)


def _panel(d, host=False):
    return torch.zeros((d.panel_h, d.panel_w, 4), dtype=torch.uint8, **(dict(pin_memory=True) if host else
                                                                         dict(device="cuda")))


def _pose(rng):
    return S.model_matrix(int(rng.integers(0, 120)))


def prepare(case, seed):
    return {"frame": _prepare_frame, "batch": _prepare_batch, "learned": _prepare_learned,
            "network": _prepare_learned, "sample": _prepare_sample}[case["kind"]](case, int(seed))


def _prepare_frame(c, seed):
    rng = np.random.default_rng(seed)
    d = S.display_tiny() if c.get("tiny") else _display(c)
    stream = torch.cuda.current_stream()
    R = lfdpr.Renderer(d, _scene(c, seed), max_points=(1 << 24) if c["ss"] else 0, stream=stream,
                       shading=S.Shading() if c.get("pbr") else None)
    held = _Held(R)
    if d.recon in (2, 3):
        R.set_view_jitter(rng.random(d.n_render_views).astype(np.float32))
        R.set_recon_samples((rng.normal(0.0, 1.0, (8, 3)) * SIGMA).astype(np.float32))
    panel = _panel(d, c.get("host", False))
    out = dict(_of_display(held, R.buffers(), d.n_render_views, d), panel=panel)
    return dict(kind="frame", renderer=R, model=_pose(rng), stream=stream, panel=panel.data_ptr(), out=out)


def _prepare_batch(c, seed):
    rng = np.random.default_rng(seed)
    stream = torch.cuda.current_stream()
    displays, scenes = [], []
    for k in range(c["scenes"]):
        # sizes spread evenly over the range (in their logarithm) whatever the seed
        f = (k + 0.5) / c["scenes"]
        tris = math.exp(math.log(c["tris_lo"]) * (1 - f) + math.log(c["tris_hi"]) * f)
        inst = max(2, min(200, int(tris / 2000)))
        w, h = [(420, 560), (640, 360)][k % 2]
        displays.append(replace(S.display_paper(), n_views=[24, 48, 96][k % 3], view_w=w, view_h=h,
                                focal_w=2.4 * w / h))
        scenes.append(_geometry(inst, max(4, int(round(math.sqrt(tris / (2.0 * inst))))), c["textures"],
                                seed * 100 + k))
    tex = lfdpr.TextureSet(_textures(c["textures"], c["max_tex"], seed), stream)
    B = lfdpr.Batch(displays, scenes, tex, max_points=[1 << 21] * c["scenes"], stream=stream)
    held = _Held(B, tex)
    out = {}
    for k, d in enumerate(displays):
        out["views%d" % k] = _of_display(held, B.buffers(k), d.n_views, d, with_keys=False)["views"]
        out["panel%d" % k] = torch.as_tensor(_Memory(held, B.panel(k), (d.panel_h, d.panel_w, 4), "|u1"),
                                             device="cuda")
    models = np.stack([_pose(rng) for _ in displays])
    return dict(kind="batch", batch=B, models=models, stream=stream, out=out)


def _prepare_learned(c, seed):
    rng = np.random.default_rng(seed)
    stream = torch.cuda.current_stream()
    w, b, nin = recon_net.load_weights()
    d_in, d_out = _display(c, n_views=nin), _display(c, n_views=4 * nin)
    src = lfdpr.Renderer(d_in, _scene(c, seed), stream=stream)
    dst = _Display(d_out)
    net = lfdpr.Recon(c["w"], c["h"], nin, w, b)
    held = _Held(net, dst, src)
    panel = _panel(d_out)
    model = _pose(rng)
    src.render(model, stream)
    out = _of_display(held, _buffers(dst.disp, src.mesh), 4 * nin, d_out, with_keys=False)
    if c["kind"] == "learned":
        out["panel"] = panel
    return dict(kind=c["kind"], src=src, dst=dst, net=net, model=model, stream=stream, panel=panel.data_ptr(), out=out)


def _prepare_sample(c, seed):
    rng = np.random.default_rng(seed)
    sc = _geometry(c["instances"], c["res"], c["textures"], seed)
    d = _display(c)
    sizes = _sizes(1024)
    wh = np.array([[sizes[k % len(sizes)]] * 2 for k in range(c["textures"])], np.uint32)
    cap = 1 << 20
    mesh = [torch.from_numpy(a).cuda() for a in (sc.xyz, sc.uv, sc.idx.view(np.int32), sc.tri_tex.view(np.int32))]
    out = dict(points=torch.zeros((cap, 4), dtype=torch.int32, device="cuda"),
               counts=torch.zeros(sc.n_tris, dtype=torch.int32, device="cuda"),
               counters=torch.zeros(4, dtype=torch.int32, device="cuda"))
    return dict(kind="sample", desc=lfdpr.desc_of(d), model=_pose(rng), mesh=mesh, n_tris=sc.n_tris, wh=wh, cap=cap,
                stream=torch.cuda.current_stream(), out=out)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(state):
    kind, stream = state["kind"], state["stream"]
    if kind == "frame":
        state["renderer"].render(state["model"], stream)
        state["renderer"].interleave(state["panel"], stream)
    elif kind == "batch":
        state["batch"].render(state["models"], stream)
    elif kind == "learned":
        state["src"].render(state["model"], stream)
        state["net"].run(state["src"].disp, state["dst"].disp, stream)
        lfdpr.lfdpr_interleave(state["dst"].disp, state["panel"], stream)
    elif kind == "network":
        state["net"].run(state["src"].disp, state["dst"].disp, stream)
    else:
        xyz, uv, idx, tri_tex = state["mesh"]
        out = state["out"]
        lfdpr.lfdpr_sample_points_noalloc(state["desc"], state["model"], xyz.data_ptr(), uv.data_ptr(),
                                          idx.data_ptr(), tri_tex.data_ptr(), state["n_tris"], state["wh"],
                                          out["points"].data_ptr(), state["cap"], out["counts"].data_ptr(),
                                          out["counters"].data_ptr(), stream)
    return state["out"]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _mesh_bytes(instances, res):
    """Vertices (position, texture coordinate) and triangles (three indices, texture id), each read once."""
    return instances * (20 * (res + 1) ** 2 + 16 * 2 * res * res)


def _network_flops(w, h, nout):
    hp, wp = recon_net.padded(h, w)
    return sum(2 * 9 * ci * co * (hp >> lv) * (wp >> lv) for ci, co, lv in recon_net.LAYERS) + 2 * 32 * 3 * nout * hp * wp


def work(case):
    """The mesh read, the depth keys and views written, the panel written. The
    texels a frame samples depend on the scene and are not counted."""
    c = case
    if c.get("tiny"):
        mesh = 2048 * (3 * 20 + 16)
    elif c["kind"] == "batch":
        mesh = px = 0
        for k in range(c["scenes"]):
            f = (k + 0.5) / c["scenes"]
            mesh += 26 * math.exp(math.log(c["tris_lo"]) * (1 - f) + math.log(c["tris_hi"]) * f)
            px += [24, 48, 96][k % 3] * [420 * 560, 640 * 360][k % 2]
        return {"bytes": mesh + 12 * px + 4 * 2560 * 1600 * c["scenes"], "flops": 0}
    else:
        mesh = _mesh_bytes(c["instances"], c["res"])
    if c["kind"] == "sample":
        return {"bytes": mesh + 4 * 2 * c["res"] ** 2 * c["instances"], "flops": 0}
    px, panel = c["w"] * c["h"], 4 * c["panel_w"] * c["panel_h"]
    if c["kind"] == "network":
        return {"bytes": 12 * px * 12 + 48 * px * 4, "flops": _network_flops(c["w"], c["h"], 48)}
    if c["kind"] == "learned":
        return {"bytes": mesh + 12 * px * 12 + 48 * px * 4 + panel, "flops": _network_flops(c["w"], c["h"], 48)}
    nr = c["views"] * (2 if c["recon"] in (1, 2) else 1)
    return {"bytes": mesh + 12 * nr * px + panel, "flops": 0}


def exact(case, seed):
    """Every output is a whole number fixed by the binary32 specification: none has a 64-bit value."""
    return None
