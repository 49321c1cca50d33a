"""The work that users of the library have it do, as cases that can be timed and compared.

A case names one use of the C ABI through its Python binding (``paper_2305_07083_gb300.dfb``):

* ``frames``:  one framebuffer; a frame, or the passes of a progressive render, with the read-back of its buffers;
* ``batch``:   the frames of several framebuffers composited together (``dfb_run_frames``), once or over the
  passes of their accumulation;
* ``noalloc``: one frame through the allocation-free call into the caller's buffers;
* ``convert``: FP32 fragment tiles to a storage format (the producer's side).

Inputs are drawn on the GPU from a seed.  The geometry of a scene (camera, bricks, so how many fragment tiles each
image tile gets) follows from the case alone (``view`` picks the camera); the seed draws the values and the arrival
order.  Scenes:

* ``bricks``:  disjoint bricks of a volume, one producer each, fragment tiles where a brick projects to; order keys
  follow the visibility order (data-parallel rendering);
* ``overlap``: the producers' domains reach into each other (particles with a radius, load-balanced partitions that
  are not convex), so that per-pixel depths are not in key order;
* ``renders``: every image tile rendered ``per_tile`` times with different seeds (image-parallel rendering; one
  render per tile is the ordinary progressive pass).

Left out is host memory as a source of tiles: that path runs at the speed of the host link, which differs by a
factor of two between passes on one machine.
"""

import math

import numpy as np
import torch

from paper_2305_07083_gb300 import dfb as D

DTYPES = {"f32": D.DFB_F32, "f16": D.DFB_F16, "bf16": D.DFB_BF16, "fp8": D.DFB_FP8E4M3}
MODES = {"depth": D.DFB_BLEND_DEPTH, "ordered": D.DFB_BLEND_ORDERED, "nearest": D.DFB_ZCOMPOSITE,
         "average": D.DFB_AVERAGE}
ELEMENT = {"f32": 4, "f16": 2, "bf16": 2, "fp8": 1}
DISTINCT = 4  # distinct passes of an accumulation kept resident; longer ones cycle through them


# ---- the cases ---------------------------------------------------------------
def listed():
    return [
        # A viewer's small interactive frame of a data-parallel render: few launches' worth of work, so latency.
        {"name": "interactive_256_f32", "kind": "frames", "W": 256, "H": 256, "T": 64, "scene": "bricks", "gx": 2,
         "gy": 2, "gz": 2, "view": 1, "mode": "depth", "dtype": "f32", "passes": 1, "submit": "arrays"},
        # Depth compositing of opaque surfaces (isosurfaces) at a display's size, one new frame each time; 1080
        # is no multiple of the tile.
        {"name": "nearest_1080p_bf16", "kind": "frames", "W": 1920, "H": 1080, "T": 64, "scene": "bricks", "gx": 4,
         "gy": 3, "gz": 3, "view": 2, "mode": "nearest", "dtype": "bf16", "passes": 1, "submit": "arrays"},
        # The benchmark's headline: a volume in 64 bricks refined over 16 passes at 2048x2048, FP32.
        {"name": "progressive_2048_f32", "kind": "frames", "W": 2048, "H": 2048, "T": 64, "scene": "bricks", "gx": 4,
         "gy": 4, "gz": 4, "view": 0, "mode": "depth", "dtype": "f32", "passes": 16, "submit": "arrays"},
        # The same render stored in FP16.
        {"name": "progressive_2048_f16", "kind": "frames", "W": 2048, "H": 2048, "T": 64, "scene": "bricks", "gx": 4,
         "gy": 4, "gz": 4, "view": 0, "mode": "depth", "dtype": "f16", "passes": 16, "submit": "arrays"},
        # The benchmark's precision form in its narrowest storage; the still camera's tiles submitted as a
        # prepared set.
        {"name": "progressive_4096_fp8", "kind": "frames", "W": 4096, "H": 1024, "T": 64, "scene": "bricks", "gx": 8,
         "gy": 4, "gz": 4, "view": 3, "mode": "depth", "dtype": "fp8", "passes": 16, "submit": "prepared"},
        # Producers with overlapping domains: most pixels need the sort, and the middle tiles have long lists.
        {"name": "overlap_1024_f32", "kind": "frames", "W": 1024, "H": 1024, "T": 64, "scene": "overlap", "gx": 4,
         "gy": 4, "gz": 4, "view": 4, "mode": "depth", "dtype": "f32", "passes": 1, "submit": "arrays"},
        # Image-parallel refinement with redundant renders (adaptive sampling); a denoiser takes the mean and the
        # variance images after every pass.
        {"name": "denoised_1080p_f32", "kind": "frames", "W": 1920, "H": 1080, "T": 64, "scene": "renders",
         "per_tile": 4, "view": 0, "mode": "average", "dtype": "f32", "passes": 4, "submit": "arrays",
         "read": "each"},
        # The benchmark's batched form: mixed frame sizes and brick counts in one launch.
        {"name": "batch_mixed_f16", "kind": "batch", "count": 16, "side": 1024, "T": 64, "scene": "bricks", "view": 5,
         "mode": "depth", "dtype": "f16", "passes": 1},
        # A server stepping progressive jobs of one opaque tile per image tile: the state is most of the bytes.
        {"name": "server_steps_f16", "kind": "batch", "count": 8, "side": 1024, "T": 64, "scene": "renders",
         "per_tile": 1, "view": 0, "mode": "depth", "dtype": "f16", "passes": 8},
        # An in-situ caller that may not allocate: list-order blending, small tiles, a ragged laptop-sized frame.
        {"name": "noalloc_1366_bf16", "kind": "noalloc", "W": 1366, "H": 768, "T": 32, "scene": "bricks", "gx": 4,
         "gy": 4, "gz": 4, "view": 6, "mode": "ordered", "dtype": "bf16"},
        # Producers storing the 2048x2048 frame's tiles in FP8 with a scale per tile.
        {"name": "convert_2048_fp8", "kind": "convert", "tiles": 5585, "T": 64, "dtype": "fp8"},
        # Producers storing a 1080p frame's tiles in FP16.
        {"name": "convert_1080p_f16", "kind": "convert", "tiles": 2313, "T": 64, "dtype": "f16"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _estimate(c):
    """Bytes of one pass from the case alone, high rather than low (fragments per pixel 1.5 times the longest grid
    axis, more where domains overlap)."""
    if c["kind"] == "convert":
        return c["tiles"] * c["T"] * c["T"] * 4 * (4 + ELEMENT[c["dtype"]])
    depth = c["per_tile"] if c["scene"] == "renders" else (
        12 if c["kind"] == "batch" else 1.5 * max(c["gx"], c["gy"], c["gz"]) + 1)
    if c["scene"] == "overlap":
        depth *= 2.5
    px = (1.5 if c["scene"] == "renders" else 2.4) * c["side"] ** 2 * c["count"] if c["kind"] == "batch" else (
        c["W"] * c["H"])
    return px * c.get("passes", 1) * (depth * (4 * ELEMENT[c["dtype"]] + 4) + 90)


def draw(rng):
    kind = rng.choice(["frames"] * 5 + ["batch"] * 2 + ["noalloc"] * 2 + ["convert"] * 2)
    T = rng.choice([16, 32, 64, 64, 64, 128])
    dtype = rng.choice(["f32", "f32", "f16", "bf16", "fp8"])
    if kind == "convert":
        return {"kind": kind, "tiles": max(1, _log(rng, 2 ** 17, 2 ** 24) // (T * T)), "T": T,
                "dtype": rng.choice(["f16", "bf16", "fp8"])}
    scene = rng.choice(["bricks", "bricks", "bricks", "overlap", "renders"])
    mode = {"bricks": rng.choice(["depth", "depth", "ordered", "nearest"]), "overlap": "depth",
            "renders": rng.choice(["average", "depth"])}[scene]
    c = {"kind": kind, "T": T, "scene": scene, "mode": mode, "dtype": dtype, "view": rng.randrange(1000)}
    if scene == "renders":
        c["per_tile"] = rng.choice([1, 1, 2, 4, 7])
    if kind == "batch":
        if scene == "overlap":
            c["scene"] = "bricks"
        c["count"] = rng.randint(2, 16)
        c["side"] = _log(rng, 150, 1024)
        c["passes"] = rng.choice([1, 2, 8])
    else:
        c["W"], c["H"] = _log(rng, 150, 4096), _log(rng, 150, 2200)
        if scene != "renders":
            g = rng.randint(2, 6 if scene == "bricks" else 5)
            c["gx"], c["gy"], c["gz"] = g, max(1, g - rng.randrange(2)), max(1, g - rng.randrange(2))
        if T < 64:  # the allocation-free call's fixed scratch, and tiles kept in proportion to the frame
            c["W"], c["H"] = min(c["W"], 45 * T), min(c["H"], 45 * T)
    if kind == "frames":
        c["passes"] = rng.choice([1, 1, 2, 5, 16])
        c["submit"] = rng.choice(["arrays", "arrays", "prepared"])
        if c["passes"] > 1 and rng.random() < 0.3:
            c["read"] = "each"
    most = _estimate(listed()[2])
    while _estimate(c) > most:
        if c.get("passes", 1) > 1:
            c["passes"] = max(1, c["passes"] // 2)
        elif kind == "batch":
            c["count"] = max(2, c["count"] // 2)
            c["side"] = c["side"] * 3 // 4
        else:
            c["W"], c["H"] = c["W"] * 3 // 4, c["H"] * 3 // 4
    return c


# ---- scenes ------------------------------------------------------------------
def _frame_specs(case):
    """The frames of a case: (W, H, grid or None, per_tile, overlap, camera number)."""
    if case["kind"] == "batch":
        s, rng, out = case["side"], np.random.default_rng([case["view"], 4]), []
        for i in range(case["count"]):
            g = int(rng.integers(2, 9))
            if case["scene"] == "renders":
                W, H = [(s, s), (2 * s, s)][i % 2]
                out.append((W, H, None, case["per_tile"], False, 0))
                continue
            W, H = [((s + 1) // 2, (s + 1) // 2), (s, s), (2 * s, 2 * s), (4 * s, s)][i % 4]
            out.append((W, H, (2 * g, g, g) if W > 2 * H and g <= 4 else (g, g, g), 0, False,
                        case["view"] * 1000 + i))
        return out
    grid = None if case["scene"] == "renders" else (case["gx"], case["gy"], case["gz"])
    return [(case["W"], case["H"], grid, case.get("per_tile", 0), case["scene"] == "overlap", case["view"])]


def _geometry(W, H, T, grid, per_tile, overlap, camera):
    """(tile ids, keys, hit, near, far): numpy arrays per fragment tile and GPU tensors per pixel of it; a scene of
    renders has no hit, near and far."""
    tiles_x, tiles_y = -(-W // T), -(-H // T)
    if grid is None:
        ids = np.tile(np.arange(tiles_x * tiles_y, dtype=np.int32), per_tile)
        return ids, np.zeros(len(ids), np.float32), None, None, None
    extent = np.array([2.0, 1.0, 1.0] if W > 2 * H else [1.0, 1.0, 1.0])
    radius = 1.6 if overlap else (1.2 if extent[0] > 1 else 1.0)
    rng = np.random.default_rng([camera, 7])
    th, el = rng.uniform(0, 2 * np.pi), rng.uniform(-0.35, 0.35)
    centre = extent / 2
    eye = centre + radius * np.array([np.cos(th) * np.cos(el), np.sin(el), np.sin(th) * np.cos(el)])
    fwd = (centre - eye) / np.linalg.norm(centre - eye)
    right = np.cross(fwd, [0.0, 1.0, 0.0])
    right /= np.linalg.norm(right)
    up = np.cross(right, fwd)
    size = extent / np.array(grid)
    lo = np.stack(np.meshgrid(*[np.arange(g) for g in grid], indexing="ij"), -1).reshape(-1, 3) * size
    hi = lo + size
    keys = np.linalg.norm((lo + hi) / 2 - eye, axis=1).astype(np.float32)
    if overlap:
        lo, hi = lo - 0.25 * size, hi + 0.25 * size
    pick = np.array([[(i >> b) & 1 for b in range(3)] for i in range(8)], bool)
    rel = np.where(pick, hi[:, None, :], lo[:, None, :]) - eye
    zc = rel @ fwd
    tan = np.tan(np.radians(60.0) / 2)
    zs = np.maximum(zc, 1e-9)
    sx = ((rel @ right) / zs / (tan * W / H) + 1) * 0.5 * W
    sy = (1 - (rel @ up) / zs / tan) * 0.5 * H
    brick, tile = [], []
    for b in range(len(lo)):
        x0, x1 = max(sx[b].min(), 0) // T, (min(np.ceil(sx[b].max()), W) - 1) // T
        y0, y1 = max(sy[b].min(), 0) // T, (min(np.ceil(sy[b].max()), H) - 1) // T
        if zc[b].min() <= 1e-6 or x1 < x0 or y1 < y0 or sx[b].max() <= 0 or sy[b].max() <= 0:
            continue
        t = np.arange(int(y0), int(y1) + 1)[:, None] * tiles_x + np.arange(int(x0), int(x1) + 1)[None, :]
        tile.append(t.reshape(-1))
        brick.append(np.full(t.size, b))
    brick = np.concatenate(brick) if brick else np.zeros(0, np.int64)
    tile = np.concatenate(tile) if tile else np.zeros(0, np.int64)
    d = lambda a: torch.as_tensor(a, device="cuda", dtype=torch.float64)  # noqa: E731
    p = torch.arange(T * T, device="cuda")
    hits, nears, fars = [], [], []
    step = max(1, (1 << 23) // (T * T))
    for i in range(0, len(tile), step):
        t, b = tile[i:i + step], brick[i:i + step]
        x = d(t % tiles_x)[:, None] * T + (p % T)
        y = d(t // tiles_x)[:, None] * T + (p // T)
        u, v = (2 * (x + 0.5) / W - 1) * tan * (W / H), (1 - 2 * (y + 0.5) / H) * tan
        near, far = torch.zeros_like(x), torch.full_like(x, math.inf)
        length = (1 + u * u + v * v).sqrt()
        for a in range(3):
            inv = length / (float(fwd[a]) + u * float(right[a]) + v * float(up[a]))
            t0, t1 = (d(lo[b, a]) - eye[a])[:, None] * inv, (d(hi[b, a]) - eye[a])[:, None] * inv
            near, far = torch.maximum(near, torch.minimum(t0, t1)), torch.minimum(far, torch.maximum(t0, t1))
        hits.append((far > near) & (x < W) & (y < H))
        nears.append(near.float())
        fars.append(far.float())
    if not hits:
        e = torch.zeros((0, T * T), device="cuda")
        return tile.astype(np.int32), keys[brick], e > 0, e, e
    hit, near, far = torch.cat(hits), torch.cat(nears), torch.cat(fars)
    keep = hit.any(1)
    k = keep.cpu().numpy()
    return tile[k].astype(np.int32), keys[brick][k], hit[keep], near[keep], far[keep]


def _store(rgba, dtype):
    """FP32 tiles in a storage format: (stored, scales or None)."""
    if dtype == "fp8":
        amax = rgba.abs().amax((1, 2))
        scale = torch.where(amax > 0, amax / 448.0, torch.ones_like(amax))
        return (rgba / scale[:, None, None]).clamp_(-448.0, 448.0).to(torch.float8_e4m3fn), scale
    return rgba.to({"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}[dtype]), None


def _frame_inputs(case, spec, gen, rng):
    """One frame's fragment tiles in arrival order: ids, keys, depth and one stored RGBA pool per distinct pass."""
    T, dtype = case["T"], case["dtype"]
    ids, keys, hit, near, far = _geometry(spec[0], spec[1], T, *spec[2:])
    n, passes = len(ids), min(case.get("passes", 1), DISTINCT)
    perm = rng.permutation(n)
    ids, keys = np.ascontiguousarray(ids[perm]), np.ascontiguousarray(keys[perm])
    rand = lambda *s: torch.rand(s, generator=gen, device="cuda")  # noqa: E731
    pools = []
    if hit is None:  # renders of an image tile: opaque, with noise from pass to pass
        depth = 1.0 + rand(n, T * T)
        for _ in range(passes):
            rgba = torch.ones((n, T * T, 4), device="cuda")
            rgba[..., :3] = rand(n, T * T, 3)
            pools.append(_store(rgba, dtype))
        return {"ids": ids, "keys": keys, "depth": depth, "pools": pools}
    at = torch.as_tensor(perm, device="cuda")
    hit, near, far = hit[at], near[at], far[at]
    depth = torch.where(hit, near + rand(n, T * T) * (far - near), torch.full_like(near, math.inf))
    if case["mode"] == "nearest":
        alpha = hit.float()
    else:  # Beta(2, 5) from gamma draws
        draws = [rand(n, T * T).clamp_min_(1e-12) for _ in range(4)]
        x = -(draws[0] * draws[1]).log()
        y = -(draws[2] * draws[3]).log()
        y -= (rand(n, T * T).clamp_min_(1e-12) * rand(n, T * T).clamp_min_(1e-12) *
              rand(n, T * T).clamp_min_(1e-12)).log()
        alpha = x / (x + y) * hit
        del draws, x, y
    del near, far, hit
    base = rand(n, T * T, 3)
    for _ in range(passes):
        rgb = base
        if passes > 1:
            rgb = (base + 0.02 * torch.randn(base.shape, generator=gen, device="cuda")).clamp_(0.0, 1.0)
        pools.append(_store(torch.cat([rgb * alpha[..., None], alpha[..., None]], -1), dtype))
    return {"ids": ids, "keys": keys, "depth": depth, "pools": pools}


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    rng = np.random.default_rng(int(seed))
    if case["kind"] == "convert":
        n, P = case["tiles"], case["T"] ** 2
        rgba = torch.rand((n, P, 4), generator=gen, device="cuda")
        alpha = rgba[..., 3:] * (torch.rand((n, P, 1), generator=gen, device="cuda") < 0.8)
        return torch.cat([rgba[..., :3] * alpha, alpha], -1)
    return [_frame_inputs(case, spec, gen, rng) for spec in _frame_specs(case)]


# ---- what a user's program keeps, and one pass -------------------------------
class _Frame:
    """A framebuffer handle with its fragment pools and the device images it is read into."""

    def __init__(self, case, spec, data):
        W, H = spec[:2]
        T, dtype = case["T"], case["dtype"]
        n, tile = len(data["ids"]), T * T * 4
        self.data = data
        self.rgba = [D.pool_pointers(p, n, tile * ELEMENT[dtype]) for p, _ in data["pools"]]
        self.scales = [None if s is None else s.cpu().numpy() for _, s in data["pools"]]
        self.depth = D.pool_pointers(data["depth"], n, tile)
        self.color = torch.empty((H, W, 4), device="cuda")
        self.rgba8 = torch.empty((H, W), dtype=torch.int32, device="cuda")
        self.handle, self.sets = None, []
        if case["kind"] == "noalloc":
            return
        self.accumulates = case["passes"] > 1
        flags = D.DFB_FLAGS_DEFAULT
        if case["kind"] == "batch":  # a server's accumulating job displays its mean and needs no image of the pass
            flags = D.DFB_FLAG_PACK_RGBA8 | (D.DFB_FLAG_ACCUMULATE if self.accumulates else D.DFB_FLAG_WRITE_COLOR)
        self.handle = D.dfb_create_ex(W, H, T, MODES[case["mode"]], DTYPES[dtype], flags, 0, n)
        if self.accumulates:
            self.mean = torch.empty((H, W, 4), device="cuda")
            self.variance = torch.empty((H, W, 4), device="cuda")
            self.tile_variance = torch.empty(-(-W // T) * -(-H // T), device="cuda")
        if case["kind"] == "batch" or case["submit"] == "prepared":
            self.sets = [D.dfb_tileset_create(self.handle, data["ids"], data["keys"], r, self.depth, s)
                         for r, s in zip(self.rgba, self.scales)]

    def __del__(self):
        for s in self.sets:
            D.dfb_tileset_destroy(s)
        if self.handle is not None:
            D.dfb_destroy(self.handle)


def prepare(case, seed):
    if case["kind"] == "convert":
        src = _inputs(case, seed)
        kind = {"f16": torch.float16, "bf16": torch.bfloat16, "fp8": torch.uint8}[case["dtype"]]
        scales = torch.empty(case["tiles"], device="cuda") if case["dtype"] == "fp8" else None
        return {"case": case, "src": src, "dst": torch.empty(src.shape, dtype=kind, device="cuda"), "scales": scales}
    return {"case": case, "frames": [_Frame(case, spec, data)
                                     for spec, data in zip(_frame_specs(case), _inputs(case, seed))]}


def _run_frames(case, f, stream):
    h, passes, each = f.handle, case["passes"], case.get("read") == "each"
    for p in range(passes):
        k = p % len(f.rgba)
        if f.sets:
            D.dfb_run_frames([h], [f.sets[k]], [int(p > 0)], stream)
        else:
            D.dfb_begin_frame(h, int(p > 0))
            D.dfb_submit_tiles(h, f.data["ids"], f.data["keys"], f.rgba[k], f.depth, f.scales[k], D.DFB_PTR_DEVICE)
            D.dfb_end_frame(h, stream)
        if each and p + 1 < passes:
            D.dfb_read_accum(h, f.mean)
            D.dfb_read_variance(h, f.variance, f.tile_variance)
    return _read(f)


def _read(f, color=True, variance=True):
    out = {"rgba8": f.rgba8}
    D.dfb_read_rgba8(f.handle, f.rgba8)
    if color:
        out["color"] = f.color
        D.dfb_read_color(f.handle, f.color)
    if f.accumulates:
        out["mean"] = f.mean
        D.dfb_read_accum(f.handle, f.mean)
        if variance:
            out["variance"], out["tile_variance"] = f.variance, f.tile_variance
            D.dfb_read_variance(f.handle, f.variance, f.tile_variance)
    return out


def run(state):
    case, stream = state["case"], torch.cuda.current_stream()
    if case["kind"] == "convert":
        D.dfb_convert_tiles(state["src"], state["dst"], state["scales"], case["tiles"], case["T"] ** 2,
                            DTYPES[case["dtype"]], stream)
        return {"tiles": state["dst"], "scales": state["scales"]}
    frames = state["frames"]
    if case["kind"] == "frames":
        return _run_frames(case, frames[0], stream)
    if case["kind"] == "noalloc":
        f = frames[0]
        D.dfb_composite_noalloc(f.color.shape[1], f.color.shape[0], case["T"], MODES[case["mode"]],
                                DTYPES[case["dtype"]], f.data["ids"], f.data["keys"], f.rgba[0], f.depth,
                                f.scales[0], None, f.color, f.rgba8, stream)
        return {"rgba8": f.rgba8, "color": f.color}
    handles = [f.handle for f in frames]
    for p in range(case["passes"]):
        D.dfb_run_frames(handles, [f.sets[p % len(f.sets)] for f in frames], [int(p > 0)] * len(frames), stream)
    return [_read(f, color=case["passes"] == 1, variance=False) for f in frames]


# ---- what a pass cannot do without -------------------------------------------
def work(case):
    if case["kind"] == "convert":
        v = case["tiles"] * case["T"] ** 2 * 4
        return {"bytes": v * (4 + ELEMENT[case["dtype"]]), "flops": v}
    nbytes = flops = 0
    passes = case.get("passes", 1)
    for spec in _frame_specs(case):
        W, H, T = spec[0], spec[1], case["T"]
        ids = _geometry(W, H, T, *spec[2:])[0]
        tiles_x = -(-W // T)
        frag = int((np.minimum(T, W - ids % tiles_x * T) * np.minimum(T, H - ids // tiles_x * T)).sum())
        px, rgba = W * H, 4 * ELEMENT[case["dtype"]]
        one = {"depth": frag * (rgba + 4), "nearest": frag * 4 + px * rgba}.get(case["mode"], frag * rgba)
        color = case["kind"] != "batch" or passes == 1
        nbytes += passes * (one + px * (20 if color else 4))  # the colour and RGBA8 images
        flops += passes * frag * 8
        if passes > 1 or case["kind"] == "frames":  # the sums and the variance state: written, then read too
            nbytes += px * 32 * (2 * passes - 1)
        if case["kind"] == "noalloc":
            continue
        last = 2 * 4 + (2 * 16 if color else 0)
        if passes > 1:
            images = 2 if case["kind"] == "frames" else 1
            last += 32 * images * (passes if case.get("read") == "each" else 1)
        nbytes += px * last  # the images read back: each read once and written once
    return {"bytes": nbytes, "flops": flops}


# ---- the same in 64 bits -----------------------------------------------------
def _decode(pool, dtype, at):
    stored, scales = pool
    v = (stored.view(torch.uint8)[at].view(stored.dtype).float() if dtype == "fp8" else stored[at]).double()
    return v * scales[at].double()[..., None, None] if scales is not None else v


def _composite64(case, spec, data, pool):
    """The frame of one pass, (H, W, 4) float64."""
    W, H, T, mode = spec[0], spec[1], case["T"], case["mode"]
    tiles_x, tiles_y = -(-W // T), -(-H // T)
    n_tiles, ids = tiles_x * tiles_y, data["ids"]
    img = torch.zeros((n_tiles, T * T, 4), dtype=torch.float64, device="cuda")
    order = np.lexsort((np.arange(len(ids)), data["keys"], ids))
    counts = np.bincount(ids, minlength=n_tiles)
    first = np.concatenate([[0], np.cumsum(counts)[:-1]])
    for n in np.unique(counts[counts > 0]):
        same = np.nonzero(counts == n)[0]
        step = max(1, (1 << 23) // (T * T * int(n)))
        for i in range(0, len(same), step):
            t = same[i:i + step]
            at = torch.as_tensor(order[first[t][:, None] + np.arange(n)], device="cuda")  # (tiles, n)
            rgba = _decode(pool, case["dtype"], at)  # (tiles, n, P, 4)
            if mode == "average":
                out = rgba.sum(1) / n
            else:
                if mode != "ordered":
                    z, by = data["depth"][at].sort(dim=1, stable=True)
                    rgba = rgba.gather(1, by[..., None].expand_as(rgba))
                if mode == "nearest":
                    out = torch.where((z[:, 0] < math.inf)[..., None], rgba[:, 0], 0.0)
                else:
                    out = torch.zeros_like(rgba[:, 0])
                    for k in range(int(n)):
                        out = out + (1.0 - out[..., 3:]) * rgba[:, k]
            img[torch.as_tensor(t, device="cuda")] = out
    img = img.reshape(tiles_y, tiles_x, T, T, 4).transpose(1, 2).reshape(tiles_y * T, tiles_x * T, 4)
    return img[:H, :W]


def exact(case, seed):
    inputs = _inputs(case, seed)
    if case["kind"] == "convert":
        if case["dtype"] != "fp8":
            return {"tiles": inputs.double(), "scales": None}
        return {"tiles": None, "scales": inputs.double().abs().amax((1, 2)) / 448.0}
    passes, out = case.get("passes", 1), []
    for spec, data in zip(_frame_specs(case), inputs):
        distinct = [_composite64(case, spec, data, p) for p in data["pools"]]
        images = [distinct[p % len(distinct)] for p in range(passes)]
        got = {"rgba8": None}
        if passes == 1 or case["kind"] == "frames":
            got["color"] = images[-1]
        if passes > 1:
            mean = sum(images[1:], images[0]) / passes
            got["mean"] = mean
            if case["kind"] == "frames":
                var = sum(((v - mean) ** 2 for v in images[1:]), (images[0] - mean) ** 2) / (passes - 1)
                got["variance"] = var
                T = case["T"]
                H, W = var.shape[:2]
                rows = torch.arange(H, device="cuda") // T
                cols = torch.arange(W, device="cuda") // T
                tile = (rows[:, None] * -(-W // T) + cols[None, :]).reshape(-1)
                sums = torch.zeros(-(-W // T) * -(-H // T), dtype=torch.float64, device="cuda")
                sums.index_add_(0, tile, var[..., :3].sum(-1).reshape(-1))
                got["tile_variance"] = sums / (3 * torch.bincount(tile, minlength=len(sums)))
        out.append(got)
    return out[0] if case["kind"] in ("frames", "noalloc") else out
