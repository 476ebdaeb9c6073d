"""Timing cases: what a program does with this library, one call per case.

Each case is a plain dict: an operation (an entry point of the package), an
image kind with its size and pixel type, and the grid edge h = h_num / h_den.
Inputs are seeded label images made on the GPU with the shapes and statistics
of the package's synthetic workloads (disks, unions of ellipses, Voronoi
labels after a 5x5 majority filter, thresholded smooth noise, stars).

Operations
  mesh        mesh_bitmap (explicit or compact format): the main call
  batch       mesh_batch over square bitmaps of mixed sizes and mixed h
  preprocess  mesh_preprocess: the moved base mesh (snap, repel, re-fan)
  embed       mesh_preprocessed: preprocessing and the retriangulation of
              every cell on the moved mesh
  project     mesh_project: a float pixel field onto a mesh at hand
  quality     mesh_quality: the quality measures of a mesh at hand
  heat        mesh_heat: diffusion steps on one label region of a mesh at hand

A program keeps one context for all its images, on its own stream, and takes
each mesh into buffers of its own (as for a renderer or a solver), sized once
for the largest mesh it expects; the unused tails stay zero.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2602_19474_gb300 as sb

# App. I's first admissible thresholds
ABC = (0.26, 0.125, 0.183)
VORONOI_LABELS = 16
VORONOI_AREA = 128 * 128  # pixels per seed, as 4096 seeds on 8192 x 8192

_context = None
_stream = None


def _ctx() -> int:
    global _context, _stream
    if _context is None:
        _stream = torch.cuda.Stream()
        _context = sb.mesh_create(0, 0, _stream.cuda_stream)
    return _context


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _case(op, image, width, height, h_num, h_den=1, dtype="u8", **more):
    return dict(op=op, image=image, width=width, height=height, h_num=h_num, h_den=h_den, dtype=dtype, **more)


def listed():
    return [
        # the smallest call: one icon-sized bitmap, where latency counts
        dict(_case("mesh", "disk", 64, 64, 2), name="disk64"),
        # a medium binary image on a coarse grid
        dict(_case("mesh", "ellipses", 2048, 2048, 4), name="ellipses2048"),
        # ragged size, grid edge far above the boundary's runs: many boundary
        # vertices per cell
        dict(_case("mesh", "noise", 1537, 1001, 8, sigma=8.0), name="noise_h8"),
        # the paper's own regime (h below one pixel): every cut cell in the table
        dict(_case("mesh", "star", 1201, 1117, 2, 3), name="star_fine"),
        # the largest: a multi-label map
        dict(_case("mesh", "voronoi", 8192, 8192, 2, dtype="u16"), name="voronoi8192"),
        # a ragged multi-label map in the compact format (for copying out)
        dict(_case("mesh", "voronoi", 5003, 3777, 2, dtype="u16", compact=True), name="voronoi_compact"),
        # one batch of a meshing service: mixed sizes, mixed h, one call
        dict(_case("batch", "noise", 256, 4096, 2, count=10, sigma=4.0), name="batch10"),
        # geometric preprocessing of the base mesh alone
        dict(_case("preprocess", "voronoi", 4096, 4096, 2, dtype="u16"), name="preprocess4096"),
        # preprocessing and retriangulation, the whole method
        dict(_case("embed", "voronoi", 4096, 4096, 2, dtype="u16"), name="embed4096"),
        # a scalar field onto the mesh: triangle means and vertex values
        dict(_case("project", "voronoi", 4096, 4096, 2, dtype="u16"), name="project4096"),
        # quality report of a mesh
        dict(_case("quality", "voronoi", 4096, 4096, 2, dtype="u16"), name="quality4096"),
        # four diffusion steps on the largest label's region
        dict(_case("heat", "voronoi", 4096, 4096, 2, dtype="u16", steps=4), name="heat4096"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["mesh", "mesh", "mesh", "batch", "preprocess", "embed", "project", "quality", "heat"])
    if op == "batch":
        lo = _log(rng, 128, 400)
        return _case("batch", "noise", lo, _log(rng, 1000, 4096), 2, count=rng.randint(2, 10), sigma=4.0)
    if op == "mesh":
        image = rng.choice(["disk", "ellipses", "noise", "star", "voronoi"])
        h = rng.choice([(2, 3), (6, 5), (2, 1), (4, 1), (8, 1)])
        if image == "star":
            h = rng.choice([(2, 3), (2, 1)])
        top = {"disk": 2048, "ellipses": 4096, "noise": 4096, "star": 2048, "voronoi": 8192}[image]
        if h[0] < 2 * h[1]:
            top = min(top, 2048)
        case = _case("mesh", image, _log(rng, 48, top), _log(rng, 48, top), *h,
                     dtype="u16" if image == "voronoi" else rng.choice(["u8", "u16"]), compact=rng.random() < 0.25)
        if image == "noise":
            case["sigma"] = round(rng.uniform(4.0, 32.0), 2)
        return case
    case = _case(op, "voronoi", _log(rng, 256, 4096), _log(rng, 256, 4096), *rng.choice([(2, 1), (2, 1), (4, 1)]),
                 dtype="u16")
    if op == "heat":
        case["steps"] = rng.randint(1, 4)
    return case


# ---------------------------------------------------------------------------
# inputs, made on the GPU from the seed alone
# ---------------------------------------------------------------------------
def _grid(h, w, x0=0.0, y0=0.0):
    y = torch.arange(h, device="cuda", dtype=torch.float32).add_(y0)[:, None]
    x = torch.arange(w, device="cuda", dtype=torch.float32).add_(x0)[None, :]
    return x, y


def _disk(rs, w, h):
    s = min(w, h)
    cx, cy = w / 2 + rs.uniform(-0.05, 0.05) * s, h / 2 + rs.uniform(-0.05, 0.05) * s
    r = s * rs.uniform(0.28, 0.36)
    x, y = _grid(h, w)
    return ((x - cx) ** 2 + (y - cy) ** 2 <= r * r).to(torch.int16)


def _ellipses(rs, w, h):
    img = torch.zeros(h, w, dtype=torch.bool, device="cuda")
    for _ in range(max(2, round(200 * w * h / 2048**2))):
        cx, cy, a, b = rs.uniform(0, w), rs.uniform(0, h), rs.uniform(10, 150), rs.uniform(10, 150)
        th, r = rs.uniform(0, math.pi), max(a, b)
        x0, x1 = max(0, int(cx - r) - 1), min(w, int(cx + r) + 2)
        y0, y1 = max(0, int(cy - r) - 1), min(h, int(cy + r) + 2)
        x, y = _grid(y1 - y0, x1 - x0, x0 - cx, y0 - cy)
        c, s = math.cos(th), math.sin(th)
        img[y0:y1, x0:x1] |= ((c * x + s * y) / a) ** 2 + ((c * y - s * x) / b) ** 2 <= 1.0
    return img.to(torch.int16)


def _noise(gen, w, h, sigma):
    z = torch.fft.rfft2(torch.randn(h, w, generator=gen, device="cuda"))
    ky = torch.fft.fftfreq(h, device="cuda")[:, None]
    kx = torch.fft.rfftfreq(w, device="cuda")[None, :]
    z[0, 0] = 0.0  # both labels in every image, however small
    z *= torch.exp(-2.0 * (math.pi * sigma) ** 2 * (kx * kx + ky * ky))
    return (torch.fft.irfft2(z, s=(h, w)) > 0).to(torch.int16)


def _star(rs, w, h):
    s, rot = min(w, h), rs.uniform(0, 2 * math.pi)
    cx, cy = w / 2 + rs.uniform(-0.03, 0.03) * s, h / 2 + rs.uniform(-0.03, 0.03) * s
    ang = rot + np.arange(10) * math.pi / 5
    rad = np.where(np.arange(10) % 2 == 0, 0.4 * s, 0.16 * s)
    px, py = cx + rad * np.cos(ang), cy + rad * np.sin(ang)
    x, y = _grid(h, w)
    inside = torch.zeros(h, w, dtype=torch.bool, device="cuda")
    for i in range(10):
        j = i - 1
        rows = (py[i] > y) != (py[j] > y)
        cross = (px[j] - px[i]) * (y - py[i]) / (py[j] - py[i]) + px[i]
        inside ^= rows & (x < cross)
    return inside.to(torch.int16)


def _voronoi(rs, w, h):
    """Labels of the nearest of uniform seeds, then a 5x5 majority filter
    (ties keep the centre label, else the smallest)."""
    n = max(4, round(w * h / VORONOI_AREA))
    sx, sy = rs.uniform(0, w, n), rs.uniform(0, h, n)
    lab = rs.randint(0, VORONOI_LABELS, n)
    tile = 256
    tx, ty = -(-w // tile), -(-h // tile)
    # per tile the seeds within 1.5 tiles of its centre, padded to one length
    near = [[np.nonzero((np.abs(sx - (i + 0.5) * tile) < 1.5 * tile) & (np.abs(sy - (j + 0.5) * tile) < 1.5 * tile))[0]
             for i in range(tx)] for j in range(ty)]
    most = max(1, max(len(v) for row in near for v in row))
    img = torch.zeros(ty * tile, tx * tile, dtype=torch.int16, device="cuda")
    x, y = _grid(tile, tile)
    for j in range(ty):
        px, py, pl = np.full((tx, most), 1e6), np.full((tx, most), 1e6), np.zeros((tx, most))
        for i in range(tx):
            k = near[j][i]
            px[i, : len(k)], py[i, : len(k)], pl[i, : len(k)] = sx[k] - i * tile, sy[k] - j * tile, lab[k]
        p = torch.tensor(np.stack([px, py, pl]), dtype=torch.float32, device="cuda")
        best = torch.full((tx, tile, tile), 1e30, device="cuda")
        own = torch.zeros((tx, tile, tile), device="cuda")
        for m in range(most):
            d = (x - p[0, :, m, None, None]) ** 2 + (y - p[1, :, m, None, None]) ** 2
            own = torch.where(d < best, p[2, :, m, None, None], own)
            best = torch.minimum(d, best)
        img[j * tile : (j + 1) * tile] = own.permute(1, 0, 2).reshape(tile, tx * tile).to(torch.int16)
    img = img[:h, :w].contiguous()
    top = torch.full((h, w), -1, dtype=torch.int16, device="cuda")
    arg, centre = torch.zeros_like(img), torch.zeros_like(img)
    for k in range(VORONOI_LABELS):
        one = torch.nn.functional.pad((img == k).to(torch.int16), (2, 2, 2, 2))
        rows = one[:, :w] + one[:, 1 : w + 1] + one[:, 2 : w + 2] + one[:, 3 : w + 3] + one[:, 4 : w + 4]
        c = rows[:h] + rows[1 : h + 1] + rows[2 : h + 2] + rows[3 : h + 3] + rows[4 : h + 4]
        centre = torch.where(img == k, c, centre)
        arg = torch.where(c > top, torch.full_like(arg, k), arg)
        top = torch.maximum(top, c)
    return torch.where(centre == top, img, arg)


def _image(case, seed):
    rs = np.random.RandomState((seed * 7919 + 104729) % (2**32))
    gen = torch.Generator(device="cuda").manual_seed(seed)
    w, h, kind = case["width"], case["height"], case["image"]
    if kind == "noise":
        img = _noise(gen, w, h, case["sigma"])
    else:
        img = {"disk": _disk, "ellipses": _ellipses, "star": _star, "voronoi": _voronoi}[kind](rs, w, h)
    return img.to(torch.uint8) if case["dtype"] == "u8" else img


def _batch_specs(case, seed):
    """(side, sigma, h) of the batch's bitmaps: sides over the logarithm of
    the range (the same ones for every seed), sigma in [4, 32], h of {2, 4, 8}."""
    rs = np.random.RandomState((seed * 6007 + 15013) % (2**32))
    n = case["count"]
    sides = np.exp(np.linspace(math.log(case["width"]), math.log(case["height"]), n)).astype(int)
    return [(int(s), float(rs.uniform(case["sigma"], 32.0)), (2, 4, 8)[k % 3]) for k, s in enumerate(sides)]


def _capacity(image, w, h, hh, sigma=8.0):
    """(vertices, triangles, cells) that the buffers of an image's mesh hold:
    twice the expected boundary, with room for the mesh's own border."""
    cells, _, _, events, inside = _counts(image, w, h, hh, sigma)
    cells = int((w + 4 * hh + 4) * (h + 4 * hh + 4) / (hh * hh * math.sqrt(3) / 4)) + 64
    more = int(2 * (events + inside)) + 8192
    return cells // 2 + int((w + h) / hh * 4) + 64 + more, cells + 2 * more, cells


def _buffers(image, w, h, hh, compact=False, sigma=8.0):
    v, t, c = _capacity(image, w, h, hh, sigma)
    shapes = {"xy": ((v, 2), torch.float64), "tri": ((t, 3), torch.int32), "label": ((t,), torch.int16),
              "code": ((t,), torch.int16)}
    if compact:
        shapes.update(cell_label=((c,), torch.int16), cell_code=((c,), torch.int16), patch_cell=((c,), torch.int32),
                      patch_off=((c + 1,), torch.int32))
    return {k: torch.zeros(s, dtype=d, device="cuda") for k, (s, d) in shapes.items()}


class _State:
    """One input, the program's buffers, and the mesh at hand where the
    operation works on one."""

    def __init__(self, case):
        self.case, self.mesh = case, None

    def __del__(self):
        try:
            if self.mesh is not None:
                sb.mesh_release(_ctx(), self.mesh)
        except Exception:
            pass


def prepare(case, seed):
    s = _State(case)
    ctx = _ctx()
    w, h, hh, op = case["width"], case["height"], case["h_num"] / case["h_den"], case["op"]
    if op == "batch":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        specs = _batch_specs(case, seed)
        s.imgs = [_noise(gen, side, side, sigma).to(torch.uint8) for side, sigma, _ in specs]
        s.h = [q for _, _, q in specs]
        s.out = [_buffers("noise", side, side, q, sigma=case["sigma"]) for side, _, q in specs]
        torch.cuda.synchronize()
        return s
    s.img = _image(case, seed)
    torch.cuda.synchronize()  # the context works on a stream of its own
    if op in ("mesh", "preprocess", "embed"):
        s.out = _buffers(case["image"], w, h, hh, case.get("compact", False), case.get("sigma", 8.0))
    else:  # a mesh at hand
        s.mesh = sb.mesh_bitmap(ctx, s.img, case["h_num"], case["h_den"])
        s.view = sb.mesh_query(ctx, s.mesh, -1)
        v, t, _ = _capacity(case["image"], w, h, hh)
    if op == "project":
        gen = torch.Generator(device="cuda").manual_seed(seed + 1)
        x, y = _grid(h, w)
        s.field = torch.sin(x / 37.0) * torch.cos(y / 53.0) + 0.1 * torch.randn(h, w, generator=gen, device="cuda")
        s.tri_value = torch.zeros(t, device="cuda")
        s.vertex_value = torch.zeros(v, device="cuda")
    if op == "heat":
        s.label = int(torch.bincount(s.img.reshape(-1).to(torch.int64)).argmax())
        s.u = torch.zeros(v, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return s


def _heat_args(case):
    """alpha, dt, steps, x0, y0, sigma as in the package's benchmark."""
    return 500.0, 0.01, case["steps"], case["width"] / 2.0, case["height"] / 2.0, 127.0


def _take(ctx, mesh, out):
    """A finished mesh into the program's buffers; its handle is released."""
    view = sb.mesh_query(ctx, mesh, -1)
    for name, t in sb.view_tensors(view).items():
        out[name][: len(t)].copy_(t, non_blocking=True)
    sb.mesh_release(ctx, mesh)
    return {**out, "n_vertices": view.n_vertices, "n_triangles": view.n_triangles}


def run(state):
    case, ctx = state.case, _ctx()
    op = case["op"]
    if op == "project":
        sb.mesh_project(ctx, state.mesh, state.field, state.tri_value, state.vertex_value)
        sb.mesh_query(ctx, state.mesh, -1)
        return {"tri_value": state.tri_value, "vertex_value": state.vertex_value}
    if op == "quality":
        return sb.mesh_quality(ctx, state.mesh)
    if op == "heat":
        u, peaks, its = sb.mesh_heat(ctx, state.mesh, state.label, *_heat_args(case), u=state.u)
        return {"u": u, "peaks": peaks, "iterations": its}
    with torch.cuda.stream(_stream):
        if op == "batch":
            meshes = sb.mesh_batch(ctx, state.imgs, state.h)
            return [_take(ctx, m, out) for m, out in zip(meshes, state.out)]
        h = case["h_num"], case["h_den"]
        if op == "mesh":
            m = sb.mesh_bitmap(ctx, state.img, *h, format=sb.SBMT_COMPACT if case.get("compact") else sb.SBMT_EXPLICIT)
        elif op == "preprocess":
            m = sb.mesh_preprocess(ctx, state.img, *h, *ABC)
        else:
            m = sb.mesh_preprocessed(ctx, state.img, *h, *ABC)
        return _take(ctx, m, state.out)


# ---------------------------------------------------------------------------
# the work of a pass
# ---------------------------------------------------------------------------
def _counts(image, w, h, hh, sigma=8.0):
    """Expected (cells, lattice vertices, cut cells, events, inside vertices)
    of an image's mesh.  The boundary's length in pixel edges follows from the
    image kind; an axis-parallel edge crosses 2 / h or 2.31 / h grid edges, and
    0.55 boundary vertices come with each pixel edge."""
    area = w * h
    cells = area / (hh * hh * math.sqrt(3) / 4)
    euclid = {
        "disk": 2.0 * min(w, h),
        "star": 2.3 * min(w, h),
        "ellipses": 0.5 * max(2, 200 * area / 2048**2) * 2 * math.pi * 80 * 0.35,
        "noise": 0.354 / sigma * area,
        "voronoi": 2.0 * area / math.sqrt(VORONOI_AREA) * (VORONOI_LABELS - 1) / VORONOI_LABELS,
    }[image]
    edges = euclid * 4 / math.pi + 2 * (w + h)
    events, inside = 2.15 / hh * edges, 0.55 * edges
    return cells, cells / 2, min(cells, events), events, inside


def _mesh_bytes(image, w, h, hh, item, compact=False, sigma=8.0):
    """The image once in, the mesh once out (16 bytes a vertex, 16 a triangle)."""
    cells, lattice, cut, events, inside = _counts(image, w, h, hh, sigma)
    if compact:
        return item * w * h + 16 * (events + inside) + 16 * (cut + 2 * events + 2 * inside) + 4 * cells + 8 * cut
    return item * w * h + 16 * (lattice + events + inside) + 16 * (cells + 2 * events + 2 * inside)


def work(case):
    op, item = case["op"], 2 if case["dtype"] == "u16" else 1
    w, h, hh = case["width"], case["height"], case["h_num"] / case["h_den"]
    sigma = case.get("sigma", 8.0)
    if op == "batch":
        return {"bytes": sum(_mesh_bytes("noise", s, s, q, 1, sigma=18.0) for s, _, q in _batch_specs(case, 0)),
                "flops": 0}
    if op == "mesh":
        return {"bytes": _mesh_bytes(case["image"], w, h, hh, item, case.get("compact", False), sigma), "flops": 0}
    cells, lattice, cut, events, inside = _counts(case["image"], w, h, hh)
    vertices, triangles = lattice + events + inside, cells + 2 * events + 2 * inside
    if op in ("preprocess", "embed"):  # the moved mesh's points replace about a third of the inside vertices
        return {"bytes": _mesh_bytes(case["image"], w, h, hh, item), "flops": 0}
    if op == "project":
        return {"bytes": 4 * w * h + 16 * vertices + 12 * triangles + 4 * (vertices + triangles), "flops": 0}
    if op == "quality":
        return {"bytes": 16 * vertices + 12 * triangles, "flops": 0}
    return {"bytes": 16 * vertices + 14 * triangles + 8 * vertices, "flops": 0}


# ---------------------------------------------------------------------------
# the values of the computed numbers in 64 bits (the mesh at hand is an input)
# ---------------------------------------------------------------------------
def _exact_means(xy, tri, field):
    """Per triangle the mean of the piecewise-constant pixel field: Green's
    theorem with F(x, y) = the field's integral along x, each edge cut at the
    pixel lines it crosses, where F is linear (the midpoint rule is exact)."""
    h, w = field.shape
    rows = torch.nn.functional.pad(field.double(), (1, 1, 1, 1))  # 0 outside the image
    pre = torch.nn.functional.pad(torch.cumsum(rows, 1), (1, 0))
    out = torch.empty(len(tri), dtype=torch.float64, device=xy.device)
    for t0 in range(0, len(tri), 1 << 20):
        p = xy[tri[t0 : t0 + (1 << 20)].long()]
        total, area = 0.0, 0.0
        for k in range(3):
            a, b = p[:, k], p[:, (k + 1) % 3]
            d = b - a
            area = area + 0.5 * (a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0])
            cuts = [torch.zeros_like(d[:, :1]), torch.ones_like(d[:, :1])]
            for ax in (0, 1):
                lo = torch.floor(torch.minimum(a[:, ax], b[:, ax]) + 0.5)
                for m in range(int(d[:, ax].abs().max()) + 2):
                    t = (lo + m + 0.5 - a[:, ax]) / torch.where(d[:, ax] == 0, torch.inf, d[:, ax])
                    cuts.append(t.clamp(0.0, 1.0)[:, None])
            t = torch.sort(torch.cat(cuts, 1), 1).values
            mid, dt = 0.5 * (t[:, 1:] + t[:, :-1]), t[:, 1:] - t[:, :-1]
            x, y = a[:, :1] + mid * d[:, :1], a[:, 1:] + mid * d[:, 1:]
            x = x.clamp(-1.0, float(w))
            c, r = torch.floor(x + 0.5).clamp(-1, w), torch.floor(y + 0.5).clamp(-1, h)
            ci, ri = c.long() + 1, r.long() + 1
            total = total + ((pre[ri, ci] + rows[ri, ci] * (x - (c - 0.5))) * dt).sum(1) * d[:, 1]
        out[t0 : t0 + (1 << 20)] = total / area
    return out


def _exact_vertices(xy, field):
    h, w = field.shape
    x, y = xy[:, 0].clamp(0, w - 1), xy[:, 1].clamp(0, h - 1)
    c, r = x.floor().clamp(max=max(w - 2, 0)), y.floor().clamp(max=max(h - 2, 0))
    u, v, ci, ri = x - c, y - r, c.long(), r.long()
    cj, rj, f = (ci + 1).clamp(max=w - 1), (ri + 1).clamp(max=h - 1), field.double()
    return ((1 - v) * ((1 - u) * f[ri, ci] + u * f[ri, cj])
            + v * ((1 - u) * f[rj, ci] + u * f[rj, cj]))


def _exact_quality(xy, tri):
    n, low, small, high, slivers, equi, s1 = len(tri), math.inf, math.inf, 0.0, 0, 0, 0.0
    areas, ratios, hist = [], [], torch.zeros(30, dtype=torch.int64, device=xy.device)
    for t0 in range(0, n, 1 << 22):
        p = xy[tri[t0 : t0 + (1 << 22)].long()]
        l2, ang = [], []
        for k in range(3):
            u, v = p[:, (k + 1) % 3] - p[:, k], p[:, (k + 2) % 3] - p[:, k]
            cross = (u[:, 0] * v[:, 1] - u[:, 1] * v[:, 0]).abs()
            ang.append(torch.rad2deg(torch.atan2(cross, (u * v).sum(1))))
            l2.append((u * u).sum(1))
        ang, l2, area = torch.stack(ang).amin(0), torch.stack(l2), 0.5 * cross
        lmax, lmin = l2.amax(0), l2.amin(0)
        low, small = min(low, float(ang.min())), min(small, float(area.min()))
        slivers += int((ang < 5.0).sum())
        equi += int((lmax - lmin <= 1e-9 * lmax).sum())
        areas.append(area)
        ratios.append(lmax / (2.0 * area))
        hist += torch.bincount((ang / 2.0).long().clamp(max=29), minlength=30)
    area, ar = torch.cat(areas), torch.cat(ratios)
    mean = float(area.mean())
    rank = torch.sort(ar).values
    return {"triangles": n, "min_angle_deg": low, "min_area": small, "slivers": slivers, "equilateral": equi,
            "area_mean": mean, "area_var": float(((area - mean) ** 2).mean()),
            "ar_median": float(rank[(n + 1) // 2 - 1]), "ar_p95": float(rank[math.ceil(0.95 * n) - 1]),
            "ar_max": float(rank[-1]), "angle_hist": [int(v) for v in hist]}


def _exact_heat(xy, tri, inside, case):
    """Backward Euler with the cotangent stiffness and the lumped mass on the
    free vertices of the region, each step by conjugate gradients to 1e-14."""
    alpha, dt, steps, x0, y0, sigma = _heat_args(case)
    nv = len(xy)
    mark = torch.zeros(nv, dtype=torch.bool, device=xy.device)
    free = mark.clone()
    free[tri[inside].long().reshape(-1)] = True
    mark[tri[~inside].long().reshape(-1)] = True
    free &= ~mark
    t = tri[inside].long()
    p = xy[t]
    mass = torch.zeros(nv, dtype=torch.float64, device=xy.device)
    ii, jj, ww = [], [], []
    for k in range(3):
        u, v = p[:, (k + 1) % 3] - p[:, k], p[:, (k + 2) % 3] - p[:, k]
        cross = (u[:, 0] * v[:, 1] - u[:, 1] * v[:, 0]).abs()
        ii.append(t[:, (k + 1) % 3])
        jj.append(t[:, (k + 2) % 3])
        ww.append(0.5 * alpha * dt * (u * v).sum(1) / cross)
        mass.index_add_(0, t[:, k], cross / 6.0)
    i, j, wgt = torch.cat(ii), torch.cat(jj), torch.cat(ww)
    diag = mass.clone().index_add_(0, i, wgt).index_add_(0, j, wgt)
    free_d = free.double()

    def times(v):
        q = diag * v
        q.index_add_(0, i, -wgt * v[j])
        q.index_add_(0, j, -wgt * v[i])
        return q * free_d

    u = torch.exp(-((xy[:, 0] - x0) ** 2 + (xy[:, 1] - y0) ** 2) / (2 * sigma * sigma)) * 100.0 * free_d
    inv = torch.where(free, 1.0 / diag, 0.0)
    peaks = []
    for _ in range(steps):
        b = mass * u * free_d
        r = b - times(u)
        z = inv * r
        d, rz, stop = z.clone(), float(r @ z), 1e-14 * float(b.norm())
        for _ in range(2000):
            if float(r.norm()) <= stop or rz == 0.0:
                break
            q = times(d)
            a = rz / float(d @ q)
            u = u + a * d
            r = r - a * q
            z = inv * r
            new = float(r @ z)
            d, rz = z + (new / rz) * d, new
        peaks.append(float(u.max()))
    return {"u": u, "peaks": peaks, "iterations": [None] * steps}


def _padded(t, like):
    return torch.nn.functional.pad(t, (0, len(like) - len(t)))


def exact(case, seed):
    op = case["op"]
    if op not in ("project", "quality", "heat"):
        return None  # whole numbers and coordinates of a mesh that only this library defines
    s = prepare(case, seed)
    t = sb.view_tensors(s.view)
    xy, tri = t["xy"], t["tri"]
    if op == "project":
        return {"tri_value": _padded(_exact_means(xy, tri, s.field), s.tri_value),
                "vertex_value": _padded(_exact_vertices(xy, s.field), s.vertex_value)}
    if op == "quality":
        return _exact_quality(xy, tri)
    found = _exact_heat(xy, tri, t["label"] == s.label, case)
    return {**found, "u": _padded(found["u"], s.u)}
