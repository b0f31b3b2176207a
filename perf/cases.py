"""The work a user of the renderer has it do, as cases that can be timed and compared.

A case is a dict of plain values. Its "kind" says which public calls one pass makes:

  frame    set_view, set_lens and one frame of a resident mesh, by hexfc_render ("render"), into pinned
           host memory ("host"), with tile capacities of the previous frame ("predicted") or without any
           allocation ("noalloc"); with "update" the per-cell quality and importance come before it
  batch    many views of several resident meshes in one hexfc_render_batch call
  quality  the three per-cell quality metrics of a resident mesh
  train    Adam steps of the tile-capacity network on the last frame's features and counts
  open     a mesh that is not resident yet: context, upload, first frame

Meshes are warped and jittered N^3 grids (the stand-ins of this repository's benchmark and tests); they are
resident and shared between the contexts of a process, as a server keeps them, except where the mesh is the
pass's own input (quality, open). Cameras, lenses, styles and weights come from the seed.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2009_06574_gb300 import hexfc, synth

MODE = {"sphere": synth.LENS_SPHERE, "screen": synth.LENS_SCREEN}


def _frame(name, n, w, h, **more):
    c = {"name": name, "kind": "frame", "n": n, "width": w, "height": h, "call": "render", "lens": "sphere",
         "full": False, "ortho": False, "update": False, "lod": 4}
    c.update(more)
    return c


def listed():
    return [
        # the smallest frame (the repository's parity workload): launches and waits are all of it
        _frame("ortho_4_256", 4, 256, 256, full=True, ortho=True, lod=1),
        # a small odd-sized frame for a caller that cannot let a library allocate
        _frame("noalloc_8_250x190", 8, 250, 190, call="noalloc", lens="screen", full=True, lod=2),
        # a mesh of the paper's grayloc size (24,389 cells) at 720p, the image in pinned host memory (a viewer)
        _frame("host_29_720p", 29, 1280, 720, call="host", full=True, lod=2),
        # the benchmark's step: quality and importance of every cell, then a 1080p frame
        _frame("step_64_1080p", 64, 1920, 1080, update=True),
        # the same frame in the paper's final look: screen lens, silhouettes, depth cue
        _frame("screen_64_1080p", 64, 1920, 1080, lens="screen", full=True, lod=3),
        # the largest: 2.1 M cells at 3840x2160
        _frame("frame_128_2160p", 128, 3840, 2160, lod=5),
        # one thumbnail of a large mesh: few tiles, very long bins, triangles of about a pixel
        _frame("thumb_96_320x180", 96, 320, 180, full=True),
        # a gallery: 48 thumbnails of three meshes in one call
        {"name": "batch_48_320x180", "kind": "batch", "meshes": "32,64,96", "views": 16, "width": 320, "height": 180,
         "lod": 4},
        # an animation with tile capacities of the frame before
        _frame("predicted_64_1080p", 64, 1920, 1080, call="predicted"),
        # the three deformation measures of a mesh of 262,144 cells
        {"name": "quality_64", "kind": "quality", "n": 64},
        # training of the capacity network between two 1080p frames
        {"name": "train_64_1080p", "kind": "train", "n": 64, "width": 1920, "height": 1080, "steps": 8},
        # a file is opened: context, upload and first 720p frame
        {"name": "open_24_720p", "kind": "open", "n": 24, "width": 1280, "height": 720, "lod": 2},
    ]


def draw(rng: random.Random):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["frame", "frame", "frame", "frame", "batch", "quality", "train", "open"])
    w = log_int(64, 2560)
    h = max(48, int(w * rng.uniform(0.5, 0.8)))
    if kind == "frame":
        call = rng.choice(["render", "render", "host", "predicted", "noalloc"])
        n = log_int(2, 96)
        if call == "noalloc":   # what fits its fixed scratch
            n, w, h = log_int(2, 8), min(w, log_int(64, 300)), min(h, 200)
        c = _frame("", n, w, h, call=call, lens=rng.choice(["sphere", "screen"]), full=rng.random() < 0.5,
                   ortho=rng.random() < 0.25, update=rng.random() < 0.25 and call != "noalloc",
                   lod=rng.randint(1, max(1, min(5, int(math.log2(n))))))
        c.pop("name")
        return c
    if kind == "batch":
        return {"kind": kind, "meshes": ",".join(str(log_int(4, 64)) for _ in range(rng.randint(1, 3))),
                "views": rng.randint(2, 12), "width": min(w, log_int(64, 800)), "height": min(h, log_int(48, 500)),
                "lod": rng.randint(1, 4)}
    if kind == "quality":
        return {"kind": kind, "n": log_int(4, 72)}
    if kind == "train":
        return {"kind": kind, "n": log_int(8, 64), "width": w, "height": h, "steps": rng.randint(1, 12)}
    return {"kind": kind, "n": log_int(2, 32), "width": w, "height": h, "lod": rng.randint(1, 4)}


# ------------------------------------------------------------------------------------------------- inputs

def _grid(n, seed):
    """A warped, jittered n^3 grid on [-0.5, 0.5]^3: vertices, cells (VTK corner order), LoD levels of the
    cells' edges (trailing zeros of the grid line's indices, the outer lines at the top level)."""
    rng = np.random.default_rng([seed, n])
    g = np.arange(n + 1) / n - 0.5
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    p = np.stack([x, y, z], axis=-1).reshape(-1, 3)
    s = np.sin(2 * np.pi * (p[:, [1, 2, 2, 0, 0, 1]] + rng.uniform(size=6)))
    p = p + 0.3 / n * (s[:, 0::2] * s[:, 1::2]) + rng.uniform(-0.1 / n, 0.1 / n, size=p.shape)
    k, j, i = (a.ravel() for a in np.meshgrid(*[np.arange(n)] * 3, indexing="ij"))
    corner = [(0, 0, 0), (1, 0, 0), (1, 1, 0), (0, 1, 0), (0, 0, 1), (1, 0, 1), (1, 1, 1), (0, 1, 1)]
    cells = np.stack([(i + a) + (n + 1) * ((j + b) + (n + 1) * (k + c)) for a, b, c in corner], axis=1)
    top = max(1, math.ceil(math.log2(n))) if n > 1 else 1
    line = np.array([top if m in (0, n) else min(top, (m & -m).bit_length() - 1) for m in range(n + 1)])
    a, b, c = [(line[v], line[v + 1]) for v in (i, j, k)]
    pairs = [(b[0], c[0]), (a[1], c[0]), (b[1], c[0]), (a[0], c[0]), (b[0], c[1]), (a[1], c[1]), (b[1], c[1]),
             (a[0], c[1]), (a[0], b[0]), (a[1], b[0]), (a[1], b[1]), (a[0], b[1])]
    levels = np.stack([np.minimum(u, v) for u, v in pairs], axis=1)
    return p.astype(np.float32), cells.astype(np.int32), levels.astype(np.uint8)


@functools.lru_cache(maxsize=None)
def _resident(n, own):
    """A context that holds the n^3 mesh, as a server keeps it; importance from the cells' quality. `own`: a
    mesh of its own for the passes that rewrite the importance."""
    verts, cells, levels = _grid(n, 100)
    r = hexfc.Renderer(0)
    return r, r.upload_mesh(verts, cells, None, levels), len(cells)


def _view(u, w, h, ortho=False):
    """A place on the benchmark's orbit, u in [0, 1)."""
    if ortho:
        az, el = math.radians(30.0 + 20.0 * u), math.radians(20.0)
        eye = (3 * math.cos(el) * math.sin(az), 3 * math.sin(el), 3 * math.cos(el) * math.cos(az))
        return synth.View(eye=eye, ortho_half_h=0.9, znear=0.5, zfar=6.0, width=w, height=h)
    return synth.orbit_view(120 * u, 120, w, h)


def _lens(u, w, h, mode="sphere"):
    if mode == "screen":
        return synth.Lens(mode=MODE[mode], center=(w * (0.35 + 0.3 * u), h * (0.6 - 0.2 * u), 0.0), radius=0.25 * h)
    return synth.lissajous_lens(120 * u, 120)


def _style(lod, full):
    s = synth.Style(w_base=2.0, lod=lod, delta=0.08, alpha_min=0.1, alpha_max=0.6, tf_hi=0.15)
    return s if full else synth.plain(s)


def _place(case, seed):
    u = random.Random(seed).random()
    w, h = case["width"], case["height"]
    return _view(u, w, h, case.get("ortho", False)), _lens(u, w, h, case.get("lens", "sphere"))


def prepare(case, seed):
    kind, s = case["kind"], {"case": case}
    if kind == "quality":
        s["r"] = hexfc.Renderer(0)
        verts, cells, levels = _grid(case["n"], seed)
        s["mesh"] = s["r"].upload_mesh(verts, cells, None, levels)
        s["out"] = torch.empty((3, len(cells)), device="cuda")
        return s
    w, h = case["width"], case["height"]
    if kind == "open":
        s["mesh"] = _grid(case["n"], seed)
        s["view"], s["lens"] = _place(case, seed)
        s["style"] = _style(case["lod"], True)
        s["out"] = torch.empty((h, w, 4), device="cuda")
        return s
    r = s["r"] = hexfc.Renderer(0)
    if kind == "batch":
        rng = random.Random(seed)
        s["items"] = []
        for n in map(int, case["meshes"].split(",")):
            src, mid, _ = _resident(n, False)
            mid = r.share_mesh(src, mid)
            for _ in range(case["views"]):
                u = rng.random()
                s["items"].append((mid, _view(u, w, h), _lens(u, w, h), _style(case["lod"], True),
                                   torch.empty((h, w, 4), device="cuda")))
        return s
    src, mid, n_cells = _resident(case["n"], bool(case.get("update")))
    s["mesh"] = r.share_mesh(src, mid)
    s["view"], s["lens"] = _place(case, seed)
    r.set_style(_style(case.get("lod", 4), case.get("full", False)))
    if kind == "train":
        out = torch.empty((h, w, 4), device="cuda")
        r.set_view(s["view"])
        r.set_lens(s["lens"])
        r.render(s["mesh"], out)
        g = np.random.default_rng(seed)
        sizes = [(256, 0.7), (64, 0.0), (4096, 0.177), (64, 0.0), (64, 0.125)]
        w0 = [g.normal(0.0, 1.0, k) * sd for k, sd in sizes] + [np.array([5.0])]
        s["weights"] = np.concatenate(w0).astype(np.float32)
        return s
    if case["call"] == "host":
        s["out"] = torch.empty((h, w, 4), pin_memory=True).numpy()
    else:
        s["out"] = torch.empty((h, w, 4), device="cuda")
    if case["call"] == "predicted":
        r.set_option(hexfc.HEXFC_OPT_PREDICTED_CAPACITY, 1)
    if case["update"]:
        s["importance"] = torch.empty(n_cells, device="cuda")
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "open":
        r = hexfc.Renderer(0)
        verts, cells, levels = s["mesh"]
        mesh = r.upload_mesh(verts, cells, None, levels)
        r.set_view(s["view"])
        r.set_lens(s["lens"])
        r.set_style(s["style"])
        r.render(mesh, s["out"])
        r.close()
        return s["out"]
    r = s["r"]
    if kind == "quality":
        for m in (hexfc.HEXFC_METRIC_SCALED_JACOBIAN, hexfc.HEXFC_METRIC_JACOBIAN_RATIO,
                  hexfc.HEXFC_METRIC_IMPORTANCE):
            r.cell_quality(s["mesh"], m, s["out"][m])
        return s["out"]
    if kind == "batch":
        r.render_batch(s["items"])
        return [it[4] for it in s["items"]]
    if kind == "train":
        r.capacity_set_weights(s["weights"])
        loss = r.capacity_train(case["steps"], lr=2e-3)
        return {"loss": np.float32(loss), "weights": r.capacity_get_weights()}
    r.set_view(s["view"])
    r.set_lens(s["lens"])
    out = {"image": s["out"]}
    if case["update"]:
        r.cell_quality(s["mesh"], hexfc.HEXFC_METRIC_IMPORTANCE, s["importance"])
        r.set_cell_importance(s["mesh"], s["importance"])
        out["importance"] = s["importance"]
    if case["call"] == "host":
        r.render_host(s["mesh"], s["out"])
    elif case["call"] == "noalloc":
        r.render_noalloc(s["mesh"], s["out"])
    else:
        r.render(s["mesh"], s["out"])
        if case["call"] == "predicted":
            r.finish()
    return out


# ---------------------------------------------------------------------------------------------------- work

def _geometry(n):
    """Faces (corners, edge levels and importances, 48 bytes) and vertices (12 bytes) of an n^3 grid."""
    return 48 * 3 * n * n * (n + 1) + 12 * (n + 1) ** 3


def _fragments(n, w, h, ortho=False):
    """Samples covered by the faces of an n^3 unit grid on the orbit: their projected areas, on average, where
    they lie inside the frame."""
    if ortho:
        return 1.6 * (n + 1) * (h / 1.8) ** 2 * min(1.0, w / h)
    return 1.57 * (n + 1) * (0.866 * h) ** 2 * 0.83 * min(1.0, w / h)


def work(case):
    kind = case["kind"]
    if kind == "quality":
        n = case["n"]
        return {"bytes": 3 * (36 * n ** 3 + 12 * (n + 1) ** 3), "flops": 3 * 360 * n ** 3}
    w, h = case["width"], case["height"]
    if kind == "train":   # per tile and step: forward and backward of 4 -> 64 -> 64 -> 1
        tiles = math.ceil(w / 16) * math.ceil(h / 16)
        return {"bytes": 2 * 4 * 4545 + case["steps"] * 20 * tiles, "flops": case["steps"] * tiles * 6 * 4416}
    if kind == "batch":
        ns = [int(n) for n in case["meshes"].split(",")]
        return {"bytes": case["views"] * sum(_geometry(n) + 16 * w * h for n in ns),
                "flops": case["views"] * 150 * sum(_fragments(n, w, h) for n in ns)}
    n = case["n"]
    b, f = _geometry(n) + 16 * w * h, 150 * _fragments(n, w, h, case.get("ortho", False))
    if kind == "open" or case["update"]:
        b, f = b + 36 * n ** 3 + 12 * (n + 1) ** 3, f + 360 * n ** 3
    return {"bytes": b, "flops": f}


# --------------------------------------------------------------------------------------------------- exact

def _det(a, b, c):
    return (a * torch.linalg.cross(b, c)).sum(-1)


def _quality(verts, cells, metric):
    """Scaled Jacobian, Jacobian ratio or importance of every cell in 64 bits."""
    p = torch.from_numpy(verts).cuda().double()[torch.from_numpy(cells).cuda().long()]
    nb = [(1, 3, 4), (2, 0, 5), (3, 1, 6), (0, 2, 7), (7, 5, 0), (4, 6, 1), (5, 7, 2), (6, 4, 3)]
    trip = [[p[:, m] - p[:, k] for m in nb[k]] for k in range(8)]
    x = [p[:, b] - p[:, a] for a, b in [(0, 1), (3, 2), (4, 5), (7, 6), (0, 3), (1, 2), (4, 7), (5, 6), (0, 4), (1, 5),
                                        (2, 6), (3, 7)]]
    trip.append([sum(x[4 * k:4 * k + 4]) for k in range(3)])
    det = torch.stack([_det(*t) for t in trip])
    size = torch.stack([t[0].norm(dim=1) * t[1].norm(dim=1) * t[2].norm(dim=1) for t in trip])
    sj = torch.where(size > 0, det / size, 0.0).amin(0)
    det[8] /= 64.0
    if metric == 0:
        return sj
    if metric == 1:
        return torch.where(det.amax(0) > 0, det.amin(0) / det.amax(0), -1.0)
    return (1.0 - sj).clamp(0.0, 1.0)


@functools.lru_cache(maxsize=1)
def _tables(n, seed):
    """Unique faces (canonical corners, edges' levels and importance, boundary) and vertex importance."""
    verts, cells, levels = _grid(n, seed)
    imp = _quality(verts, cells, 2)
    c = torch.from_numpy(cells).cuda().long()
    quads = [(0, 1, 2, 3), (4, 5, 6, 7), (0, 1, 5, 4), (1, 2, 6, 5), (2, 3, 7, 6), (3, 0, 4, 7)]
    q = torch.cat([c[:, list(f)] for f in quads])
    s = q.sort(dim=1).values
    order = torch.sort((s[:, 2] << 32) | s[:, 3], stable=True).indices
    order = order[torch.sort(((s[:, 0] << 32) | s[:, 1])[order], stable=True).indices]
    s, q = s[order], q[order]
    first = torch.ones(len(s), dtype=torch.bool, device="cuda")
    first[1:] = (s[1:] != s[:-1]).any(1)
    at = torch.nonzero(first)[:, 0]
    shared = torch.diff(torch.cat([at, at.new_tensor([len(s)])]))
    q = q[at]
    m = q.argmin(1)
    fwd = q.gather(1, ((m + 1) & 3)[:, None]) < q.gather(1, ((m + 3) & 3)[:, None])
    k = torch.arange(4, device="cuda")
    q = q.gather(1, torch.where(fwd, (m[:, None] + k) & 3, (m[:, None] - k) & 3))
    ends = [(0, 1), (1, 2), (2, 3), (3, 0), (4, 5), (5, 6), (6, 7), (7, 4), (0, 4), (1, 5), (2, 6), (3, 7)]
    pair = torch.stack([(torch.minimum(c[:, a], c[:, b]) << 32) | torch.maximum(c[:, a], c[:, b]) for a, b in ends], 1)
    edge, inv = pair.flatten().unique(return_inverse=True)
    lev = torch.zeros(len(edge), dtype=torch.long, device="cuda")
    lev.scatter_reduce_(0, inv, torch.from_numpy(levels).cuda().long().flatten(), "amax")
    attr = torch.zeros(len(edge), dtype=torch.double, device="cuda")
    attr.scatter_reduce_(0, inv, imp.repeat_interleave(12), "amax")
    vimp = torch.zeros(len(verts), dtype=torch.double, device="cuda")
    vimp.scatter_reduce_(0, c.flatten(), imp.repeat_interleave(8), "amax")
    nx = q.roll(-1, 1)
    fe = torch.searchsorted(edge, (torch.minimum(q, nx) << 32) | torch.maximum(q, nx))
    return torch.from_numpy(verts).cuda().double(), q, lev[fe], attr[fe], shared == 1, vimp


def _f32(x):
    return float(np.float32(x))


def _image(n, seed, view, lens, style, budget=24_000_000):
    """The frame in 64 bits: window positions on 1/256 pixel and depths of 24 bits as the renderer defines
    them, coverage and depth in integers, Eqs. 1-4, the list of every pixel in order, blended front to back."""
    P, quad, lev, attr, bound, vimp = _tables(n, seed)
    W, H = view.width, view.height
    F = [b - a for a, b in zip(view.eye, view.target)]
    zref = math.sqrt(F[0] * F[0] + F[1] * F[1] + F[2] * F[2])
    F = [v / zref for v in F]
    R = [F[1] * view.up[2] - F[2] * view.up[1], F[2] * view.up[0] - F[0] * view.up[2],
         F[0] * view.up[1] - F[1] * view.up[0]]
    rl = math.sqrt(R[0] * R[0] + R[1] * R[1] + R[2] * R[2])
    R = [v / rl for v in R]
    U = [R[1] * F[2] - R[2] * F[1], R[2] * F[0] - R[0] * F[2], R[0] * F[1] - R[1] * F[0]]
    d = [P[:, k] - view.eye[k] for k in range(3)]
    ex, ey, ed = (d[0] * B[0] + d[1] * B[1] + d[2] * B[2] for B in (R, U, F))
    ortho = not view.fovy_deg > 0
    if ortho:
        sc = (H * 0.5) / view.ortho_half_h
        xw, yw, z = W * 0.5 + ex * sc, H * 0.5 - ey * sc, (ed - view.znear) / (view.zfar - view.znear)
    else:
        fl = (H * 0.5) / math.tan(view.fovy_deg * (math.pi / 180.0) * 0.5)
        xw, yw = W * 0.5 + (ex / ed) * fl, H * 0.5 - (ey / ed) * fl
        z = (view.zfar / (view.zfar - view.znear)) * (1.0 - view.znear / ed)
    ok = (ed > view.znear) & (ed < view.zfar) & (xw.abs() <= 16384) & (yw.abs() <= 16384)
    X, Y = (xw * 256.0).round().long(), (yw * 256.0).round().long()
    Z = (z.clamp(0.0, 1.0) * 16777215.0).round().long()
    # triangles, wound to positive area: id 2 face + t
    tri = torch.stack([quad[:, [0, 1, 2]], quad[:, [0, 2, 3]]], 1).reshape(-1, 3)
    x, y = X[tri], Y[tri]
    area = (x[:, 1] - x[:, 0]) * (y[:, 2] - y[:, 0]) - (y[:, 1] - y[:, 0]) * (x[:, 2] - x[:, 0])
    tri = torch.where((area < 0)[:, None], tri[:, [0, 2, 1]], tri)
    x, y, area = X[tri], Y[tri], area.abs()
    up = lambda v: -((128 - v) // 256)  # noqa: E731  first centre at or after v (1/256 pixel)
    x0, x1 = up(x.amin(1)).clamp(min=0), ((x.amax(1) - 128) // 256).clamp(max=W - 1)
    y0, y1 = up(y.amin(1)).clamp(min=0), ((y.amax(1) - 128) // 256).clamp(max=H - 1)
    good = ok[tri].all(1) & (area > 0) & (x0 <= x1) & (y0 <= y1)
    out = torch.empty((H, W, 4), dtype=torch.double, device="cuda")
    zsil = torch.full((H * W,), 1 << 40, device="cuda", dtype=torch.long)
    bg = torch.tensor(style.bg, dtype=torch.double, device="cuda")
    total = int(((x1 - x0 + 1) * (y1 - y0 + 1))[good].sum()) if bool(good.any()) else 0
    bands = max(1, math.ceil(total / budget))
    step = max(1, H // bands)
    for r0 in range(0, H, step):
        r1 = min(H, r0 + step)
        t = torch.nonzero(good & (y1 >= r0) & (y0 < r1))[:, 0]
        b0, b1 = y0[t].clamp(min=r0), y1[t].clamp(max=r1 - 1)
        bw = x1[t] - x0[t] + 1
        cnt = bw * (b1 - b0 + 1)
        i = torch.repeat_interleave(torch.arange(len(t), device="cuda"), cnt)
        k = torch.arange(len(i), device="cuda") - (cnt.cumsum(0) - cnt)[i]
        px, py, f = x0[t][i] + k % bw[i], b0[i] + k // bw[i], t[i]
        sx, sy = 256 * px + 128, 256 * py + 128
        keep, l = torch.ones_like(px, dtype=torch.bool), []
        for e in range(3):
            a, b = (e + 1) % 3, (e + 2) % 3
            dx, dy = (x[:, b] - x[:, a])[f], (y[:, b] - y[:, a])[f]
            v = dx * (sy - y[:, a][f]) - dy * (sx - x[:, a][f])
            keep &= (v > 0) | ((v == 0) & ((dy < 0) | ((dy == 0) & (dx > 0))))
            l.append(v)
        px, py, f, sx, sy = px[keep], py[keep], f[keep], sx[keep], sy[keep]
        l1, l2, A = l[1][keep], l[2][keep], area[f]
        z0, z1, z2 = (Z[tri[:, v]][f] for v in range(3))
        zs = z0 + torch.div(l1 * (z1 - z0) + l2 * (z2 - z0), A, rounding_mode="floor")
        face = f >> 1
        if style.sil_alpha > 0:
            s = bound[face]
            zsil.scatter_reduce_(0, (py * W + px)[s], zs[s], "amin")
        rgba = _shade(sx, sy, px, py, f, face, l1.double() / A, l2.double() / A, P, quad, X, Y, lev, attr, vimp, tri, ed,
                      ortho, zref, lens, style)
        pix = (py - r0) * W + px
        order = torch.sort((pix << 24) | zs, stable=True).indices   # equal depths stay in the triangles' order
        pix, rgba = pix[order], rgba[order]
        cnt = torch.bincount(pix, minlength=(r1 - r0) * W)
        off = cnt.cumsum(0) - cnt
        c = torch.zeros((len(cnt), 3), dtype=torch.double, device="cuda")
        T = torch.ones(len(cnt), dtype=torch.double, device="cuda")
        for k in range(int(cnt.max())):
            at = torch.nonzero(cnt > k)[:, 0]
            s = rgba[off[at] + k]
            c[at] += T[at, None] * s[:, :3]
            T[at] *= 1.0 - s[:, 3]
        out[r0:r1] = torch.cat([c + T[:, None] * bg, 1.0 - T[:, None]], 1).view(r1 - r0, W, 4)
    if style.sil_alpha > 0:
        D = torch.nn.functional.pad(zsil.view(H, W), (1, 1, 1, 1), value=-1)   # -1: outside the frame
        none = 1 << 40
        mid, sil = D[1:-1, 1:-1], torch.zeros((H, W), dtype=torch.bool, device="cuda")
        side = [D[1:-1, 2:], D[1:-1, :-2], D[2:, 1:-1], D[:-2, 1:-1]]
        T = int(style.sil_threshold)
        for k, a in enumerate(side):
            b = side[k ^ 1]
            both = (a >= 0) & (a != none) & (b >= 0) & (b != none)
            sil |= (a == none) | (both & (a - mid > T) & ((a - 2 * mid + b).abs() > T))
        sil &= mid != none
        out = torch.where(sil[..., None], out + _f32(style.sil_alpha) * (1.0 - out), out)
    return out


def _shade(sx, sy, px, py, f, face, w1, w2, P, quad, X, Y, lev, attr, vimp, tri, ed, ortho, zref, lens, style):
    """Premultiplied colour and opacity (Eqs. 1-4) of the samples (sx, sy) of triangles f."""
    w0 = 1.0 - w1 - w2
    v = [tri[:, k][f] for k in range(3)]
    q = [w if ortho else w / ed[i] for w, i in zip((w0, w1, w2), v)]
    Q = q[0] + q[1] + q[2]
    imp = (q[0] * vimp[v[0]] + q[1] * vimp[v[1]] + q[2] * vimp[v[2]]) / Q
    g = torch.ones_like(Q) if ortho else (zref * Q).clamp(_f32(style.g_min), _f32(style.g_max))
    if lens.mode == synth.LENS_SCREEN:
        dist = torch.hypot(px + 0.5 - lens.center[0], py + 0.5 - lens.center[1]) / lens.radius
    else:
        at = sum(a[:, None] * P[i] for a, i in zip(q, v)) / Q[:, None]
        dist = (at - torch.tensor(lens.center, dtype=torch.double, device="cuda")).norm(dim=1) / lens.radius
    t = ((dist - 0.7) / 0.3).clamp(0.0, 1.0)
    focus = 1.0 - t * t * (3.0 - 2.0 * t)
    inf = torch.full_like(Q, math.inf)
    d_a, d_f, d_c = inf.clone(), inf.clone(), inf.clone()
    for k in range(4):
        a, b = quad[:, k][face], quad[:, (k + 1) & 3][face]
        ux, uy, ex, ey = sx - X[a], sy - Y[a], X[b] - X[a], Y[b] - Y[a]
        len2, dot = ex * ex + ey * ey, ux * ex + uy * ey
        near = torch.hypot(ux.double(), uy.double())
        far = torch.hypot((ux - ex).double(), (uy - ey).double())
        line = (ux * ey - uy * ex).abs().double() / len2.double().sqrt()
        dk = torch.where((len2 == 0) | (dot <= 0), near, torch.where(dot >= len2, far, line)) / 256.0
        ctx = lev[:, k][face] >= style.lod
        foc = ctx | (attr[:, k][face] >= _f32(style.delta))
        d_a = torch.minimum(d_a, dk)
        d_f = torch.where(foc, torch.minimum(d_f, dk), d_f)
        d_c = torch.where(ctx, torch.minimum(d_c, dk), d_c)
    wb = _f32(style.w_base)
    w = (1.0 + 0.3 * focus) * wb * g
    hw = _f32(style.halo_scale) * wb * focus * g
    e_f, e_c = (d_f <= w).double(), (d_c <= w).double()
    halo = (d_f > w) & (d_f <= w + hw) & (focus > 0)
    a_e = torch.where(halo, focus, e_c + focus * (e_f - e_c))
    tt = ((imp - _f32(style.tf_lo)) / (_f32(style.tf_hi) - _f32(style.tf_lo))).clamp(0.0, 1.0)
    s_e = torch.where(d_a <= 2.0 / 3.0 * wb, _f32(style.s), 1.0)
    a_f = _f32(style.alpha_min) + (_f32(style.alpha_max) - _f32(style.alpha_min)) * tt
    a_f = (s_e * a_f * dist.clamp(max=1.0) ** 4).clamp(max=1.0)
    beta, dark = (s_e > 1.0) * _f32(style.accent_beta), 1.0 - _f32(style.darken) * focus
    table = torch.stack([tt, torch.zeros_like(tt), 1.0 - tt], 1)
    c_e = torch.where(halo[:, None], 1.0, table * dark[:, None])
    c_f = table + beta[:, None] * (1.0 - table)
    rgb = a_e[:, None] * c_e + ((1.0 - a_e) * a_f)[:, None] * c_f
    if style.desat > 0:
        kd = (_f32(style.desat) * focus * (1.0 - g).clamp(0.0, 1.0))[:, None]
        rgb = rgb + kd * ((rgb @ rgb.new_tensor([0.299, 0.587, 0.114]))[:, None] - rgb)
    return torch.cat([rgb, (a_e + (1.0 - a_e) * a_f)[:, None]], 1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":   # a result of many rounded steps
        return None
    if kind == "quality":
        verts, cells, _ = _grid(case["n"], seed)
        return torch.stack([_quality(verts, cells, m) for m in range(3)])
    w, h = case["width"], case["height"]
    if kind == "open":
        return _image(case["n"], seed, *_place(case, seed), _style(case["lod"], True))
    if kind == "batch":
        rng, style, out = random.Random(seed), _style(case["lod"], True), []
        for n in map(int, case["meshes"].split(",")):
            for _ in range(case["views"]):
                u = rng.random()
                out.append(_image(n, 100, _view(u, w, h), _lens(u, w, h), style))
        return out
    out = {"image": _image(case["n"], 100, *_place(case, seed), _style(case["lod"], case["full"]))}
    if case["update"]:
        verts, cells, _ = _grid(case["n"], 100)
        out["importance"] = _quality(verts, cells, 2)
    return out
