"""The work that a user of this library has it do, as cases that can be timed.

Every case goes through the public binding: worlds are created, edited and
rendered by the calls a program makes.  A case is a dict of plain values:

  kind      what is called (see `run`)
  W, H      the grid; slabs: fraction of cells with a second interval;
            walls: one-cell ridges; pairs: the 2-byte paired-texel world
  w, h, n   image size and number of views
  pose      how the views are placed (see `_views`)
  shadows   one shadow ray per hit
  tile_w, tile_h, mip   render options (0, 0, -1: the library's defaults)

The terrain is seeded value noise in the shape of the paper's levels, made on
the GPU; poses are seeded too, so another seed is another world and other views.
"""

import math

import numpy as np
import torch

import paper_2608_17390_gb300 as hf

DEFAULTS = dict(slabs=0.3, walls=0, pairs=False, n=1, pose="fly", shadows=False,
                tile_w=0, tile_h=0, mip=-1)

SUN_DAY = ((300000, 120000, 200000), (-110000, -380000, 300000))


def listed():
    return [
        # A thumbnail or preview of a small level: launches and latency count.
        dict(name="thumbnail", kind="render", W=256, H=256, slabs=0.25, w=320, h=240,
             pose="oblique"),
        # The interactive player's view: one 1080p frame at eye level with shadows.
        dict(name="eye_1080p", kind="render", W=2048, H=2048, slabs=0.4, walls=512, w=1920,
             h=1080, pose="eye", shadows=True),
        # An explosion and the frame that shows it, on a level of odd size: the
        # edit-to-visible latency of the paper's dynamic-edit protocol.
        dict(name="crater_and_view", kind="edit", W=1999, H=1501, slabs=0.4, walls=300, w=641,
             h=359, pose="fly", shadows=True, edit_w=61, edit_h=57),
        # The benchmark's batch: 64 cameras from 640x360 to 4K, oblique and eye
        # level, shadows, a crater before each batch, in a tuned launch.
        dict(name="batch_64", kind="edit", W=2048, H=2048, slabs=0.4, walls=512, w=3840, h=2160,
             n=64, pose="mixed", shadows=True, edit_w=64, edit_h=64, tile_w=4, tile_h=64, mip=5),
        # A fly-through of the large level rendered a hundred frames at a time.
        dict(name="flythrough", kind="render", W=2048, H=16384, w=1920, h=1080, n=100),
        # The same level in the paper's 2-byte texels, a quarter as many frames.
        dict(name="flythrough_pairs", kind="render", W=2048, H=16384, pairs=True, w=1920, h=1080,
             n=25),
        # A moving sun: every frame asks for shadows toward another direction.
        dict(name="moving_sun", kind="suns", W=2048, H=2048, slabs=0.4, walls=512, w=1920, h=1080,
             pose="oblique", shadows=True),
        # The paper's protocol, twelve views, with its fixed-step march ...
        dict(name="march_views", kind="march", W=2048, H=16384, w=1280, h=800, n=12,
             pose="protocol", steps=128),
        # ... its atomic scatter ...
        dict(name="scatter_views", kind="scatter", W=2048, H=16384, w=1280, h=800, n=12,
             pose="protocol", nu=1024, nv=1024, nz=16),
        # ... and its voxel-accelerated march.
        dict(name="voxel_views", kind="voxel", W=2048, H=16384, w=1280, h=800, n=12,
             pose="protocol", vx=4, vy=8, vz=2, inner=4),
        # Loading a level for that renderer: the occupancy is baked, then one view.
        dict(name="voxel_bake", kind="bake", W=2048, H=16384, w=1280, h=800, pose="protocol", vx=4,
             vy=8, vz=2, inner=4),
        # A burst at the server: forty renders of 640x360 to 4K with four
        # craters between them, the craters filled again at the end.
        dict(name="serve_burst", kind="serve", W=2048, H=16384, w=3840, h=2160, n=40,
             edit_w=64, edit_h=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "edit", "edit", "suns", "march", "scatter",
                       "voxel", "bake", "serve"])
    W, H = _log_int(rng, 200, 2048), _log_int(rng, 200, 8192)
    c = dict(kind=kind, W=W, H=H, slabs=round(rng.uniform(0.0, 0.5), 2),
             walls=rng.choice([0, W * H // 8192]))
    c["w"], c["h"] = _log_int(rng, 160, 3840), _log_int(rng, 120, 2160)
    if kind == "render":
        c["pairs"] = rng.random() < 0.3
        c["W"] = W & ~1 if c["pairs"] else W
        c["n"] = rng.choice([1, 1, _log_int(rng, 2, 20)])
        c["pose"] = rng.choice(["fly", "eye", "oblique"])
        c["shadows"] = rng.random() < 0.5
        if rng.random() < 0.3:
            c["tile_w"], c["tile_h"] = rng.choice([(8, 8), (4, 32), (8, 16), (16, 4)])
            c["mip"] = rng.randint(3, 9)
    elif kind == "edit":
        c["n"] = rng.choice([1, _log_int(rng, 2, 12)])
        c["pose"] = rng.choice(["fly", "eye", "mixed"])
        c["shadows"] = rng.random() < 0.7
        c["edit_w"], c["edit_h"] = _log_int(rng, 1, 160), _log_int(rng, 1, 160)
    elif kind == "suns":
        c["pose"] = rng.choice(["fly", "oblique"])
        c["shadows"] = True
    elif kind == "serve":
        c["n"] = rng.randint(4, 40)
        c["edit_w"] = c["edit_h"] = _log_int(rng, 8, 100)
        c["shadows"] = rng.random() < 0.3
    else:
        c["pose"] = "protocol"
        c["n"] = 1 if kind == "bake" else rng.randint(1, 12)
        if kind == "march":
            c["steps"] = _log_int(rng, 16, 256)
        elif kind == "scatter":
            c["nu"], c["nv"], c["nz"] = _log_int(rng, 256, 2048), _log_int(rng, 256, 2048), \
                _log_int(rng, 4, 32)
        else:
            c["vx"], c["vy"], c["vz"] = rng.choice([(4, 8, 2), (2, 4, 1), (4, 4, 4), (3, 5, 2)])
            c["inner"] = rng.choice([4, 16])
    return c


# ------------------------------------------------------------------ inputs

def _noise(W, H, period, gen):
    """Value noise in [0, 1): four octaves, smoothstep-bilinear, on the GPU."""
    acc = torch.zeros(H, W, device="cuda")
    for o in range(4):
        p = period >> o
        lat = torch.rand(H // p + 2, W // p + 2, generator=gen, device="cuda")

        def axis(n):
            i = torch.arange(n, device="cuda")
            f = ((i % p) + 0.5) / p
            return i // p, f * f * (3 - 2 * f)

        ix, sx = axis(W)
        iy, sy = axis(H)
        rows = lat[:, ix] * (1 - sx) + lat[:, ix + 1] * sx
        acc += (rows[iy] * (1 - sy)[:, None] + rows[iy + 1] * sy[:, None]) * (0.5 ** o / 1.875)
    return acc


def _terrain(c, seed):
    """Cell words, uint32 [H, W] on the host."""
    W, H = c["W"], c["H"]
    gen = torch.Generator("cuda").manual_seed(seed)
    h0 = 20 + torch.floor(100 * _noise(W, H, 128, gen) + 0.5).int()
    m = _noise(W, H, 64, gen)
    r = torch.randint(0, 1 << 30, (H, W), generator=gen, device="cuda", dtype=torch.int32)
    mat = r & 7
    h1 = torch.clamp(h0 + 8 + (r >> 3) % 33, max=255)
    h2 = torch.clamp(h1 + 4 + (r >> 16) % 27, max=255)
    sample = m.flatten()[:: max(1, W * H // 1000000)]
    slab = m >= torch.quantile(sample, 1.0 - c["slabs"]) if c["slabs"] > 0 else m > 2
    rs = np.random.RandomState(seed % (1 << 31))
    for _ in range(c["walls"]):
        n, x, y = rs.randint(16, 257), rs.randint(1, W - 1), rs.randint(1, H - 1)
        if rs.randint(2):
            h0[y:y + n, x - 1:x + 2], slab[y:y + n, x - 1:x + 2] = 0, False
            h0[y:y + n, x] = 200
        else:
            h0[y - 1:y + 2, x:x + n], slab[y - 1:y + 2, x:x + n] = 0, False
            h0[y, x:x + n] = 200
    if c["pairs"]:  # both cells of a pair carry the same column where one has a slab
        two = slab[:, 0::2] | slab[:, 1::2]
        for v in (h0, h1, h2):
            v[:, 1::2] = torch.where(two, v[:, 0::2], v[:, 1::2])
        slab = two.repeat_interleave(2, 1)
    word = h0 | torch.where(slab, (h1 << 8) | (h2 << 16), 0) | (mat << 24)
    return word.cpu().numpy().view(np.uint32)


def _texels(cells):
    """The paired-texel form of a grid made with pairs."""
    c = cells.astype(np.uint32)
    h0, h1, h2, mat = c & 255, (c >> 8) & 255, (c >> 16) & 255, c >> 24
    slab = h1 > h0
    delta = h2 - h1
    odd = (np.arange(c.shape[1]) & 1).astype(bool)[None, :]
    nib = np.where(odd, delta & 15, delta >> 4)
    v = np.where(slab & odd, h2, h0)
    return (v | ((mat | np.where(slab, 128 | (nib << 3), 0)) << 8)).astype(np.uint16)


def _top(word):
    h0, h1, h2 = word & 255, (word >> 8) & 255, (word >> 16) & 255
    return h2 if h1 > h0 else h0


def _views(c, cells, seed):
    """Camera records.  fly: 3-50 above the terrain, looking ahead and down;
    eye: 2 above the floor, level; oblique: from above; mixed: alternating eye
    and oblique views from w x h down to a sixth of it; protocol: pitch 0, -30,
    -60, -90 at 6, 60, 120, 200 units above the terrain; path: along the grid."""
    rs = np.random.RandomState((seed * 7 + 1) % (1 << 31))
    H, W = cells.shape
    n, w, h = c["n"], c["w"], c["h"]
    cams = []
    y_path = rs.uniform(0.1, 0.3)
    for i in range(n):
        x, y, yaw = rs.uniform(2, W - 2), rs.uniform(2, H - 2), rs.uniform(0, 360)
        u, v = rs.uniform(), rs.uniform()
        pose, wi, hi, fov = c["pose"], w, h, 60 + 30 * v
        if pose == "mixed":
            pose = "eye" if i % 2 else "oblique"
            k = 1 if 4 * i < n else 2 if 8 * i < 5 * n else 6
            wi, hi = max(1, w // k), max(1, h // k)
        if pose == "fly" and n > 1:  # frames along the level
            s = i / n
            x = W * (0.5 + 0.35 * math.sin(5 * s + 6 * y_path))
            y = H * (y_path + (0.65 * s))
            yaw, u = 40 * math.cos(5 * s), 0.5 + 0.5 * math.sin(9 * s)
        word = int(cells[int(y), int(x)])
        if pose == "eye":
            while not 0 < (word & 255) < 200:
                x, y = rs.uniform(2, W - 2), rs.uniform(2, H - 2)
                word = int(cells[int(y), int(x)])
            z, pitch = (word & 255) + 2.0, -5 + 10 * u
        elif pose == "oblique":
            z, pitch = 150 + 150 * u, -80 + 50 * rs.uniform()
        elif pose == "protocol":
            k = i * 4 // n
            z, pitch, fov = _top(word) + (6, 60, 120, 200)[k], (0, -30, -60, -90)[k], 75
        else:
            z, pitch, fov = _top(word) + 3 + 47 * u, -10, 90
        cams.append(hf.hf_camera_from_pose(x, y, z, yaw, pitch, fov, wi, hi))
    return np.array(cams)


def _crater(cells, x0, y0, w, h):
    """A bowl in the rectangle: floors lowered, slabs removed in its middle."""
    b = cells[y0:y0 + h, x0:x0 + w].copy()
    yy, xx = np.mgrid[0:h, 0:w]
    r2 = ((xx - w / 2) / (w / 2)) ** 2 + ((yy - h / 2) / (h / 2)) ** 2
    drop = np.maximum(0, 40 * (1 - r2)).astype(np.int64)
    low = np.maximum(0, (b & 255).astype(np.int64) - drop).astype(np.uint32)
    b = (b & np.uint32(0xFFFFFF00)) | low
    return np.where(r2 < 0.4, b & np.uint32(0xFF0000FF), b).astype(np.uint32)


class _World:
    """A context, destroyed with the state that holds it."""

    def __init__(self, c, cells):
        self.handle = hf.hf_create_pairs(_texels(cells)) if c["pairs"] else hf.hf_create(cells)

    def __del__(self):
        hf.hf_destroy(self.handle)


def _outputs(cams, fields):
    """One block per field for all views, and each view's slices of them."""
    kinds = dict(hit_cell=torch.int32, layer=torch.uint8, face=torch.uint8, depth=torch.float32,
                 rgba=torch.int32, shadow=torch.uint8)
    px = [int(k["w"]) * int(k["h"]) for k in cams]
    blocks = {f: torch.zeros(sum(px), dtype=kinds[f], device="cuda") for f in fields}
    views = [dict() for _ in px]
    for f, t in blocks.items():
        for v, part in zip(views, t.split(px)):
            v[f] = part
    return blocks, views


def _serve_cams(c, cells, seed):
    sizes = [(c["w"], c["h"]), (c["w"] // 2, c["h"] // 2), (c["w"] // 3, c["h"] // 3),
             (c["w"] // 6, c["h"] // 6)]
    out = []
    for i in range(c["n"]):
        w, h = sizes[i % 4]
        one = dict(c, n=1, pose="fly", w=max(1, w), h=max(1, h))
        out.append(_views(one, cells, seed + 1000 * i)[0])
    return np.array(out)


def _rects(c, seed, n):
    rs = np.random.RandomState((seed * 3 + 2) % (1 << 31))
    w, h = min(c["edit_w"], c["W"]), min(c["edit_h"], c["H"])
    return [(rs.randint(0, c["W"] - w + 1), rs.randint(0, c["H"] - h + 1), w, h) for _ in range(n)]


def _inputs(case, seed):
    """The case with defaults, its cells, views and edits."""
    c = {**DEFAULTS, **case}
    cells = _terrain(c, seed)
    cams = (_serve_cams if c["kind"] == "serve" else _views)(c, cells, seed)
    edits = [(x, y, _crater(cells, x, y, w, h)) for x, y, w, h in
             (_rects(c, seed, 4 if c["kind"] == "serve" else 1) if "edit_w" in c else [])]
    return c, cells, cams, edits


def prepare(case, seed):
    c, cells, cams, edits = _inputs(case, seed)
    s = dict(kind=c["kind"], world=_World(c, cells), cams=cams, edits=edits)
    ctx = s["world"].handle
    fields = ["hit_cell", "layer", "depth"]
    if c["kind"] not in ("march", "voxel", "bake"):
        fields += ["face", "rgba"] + (["shadow"] if c["shadows"] else [])
    opts = dict(tile_w=c["tile_w"], tile_h=c["tile_h"], flags=hf.HF_SHADOWS if c["shadows"] else 0,
                mip_start=hf.HF_MIP_AUTO if c["mip"] < 0 else c["mip"])
    if c["kind"] == "suns":  # morning and afternoon, each with outputs of its own
        s["opts"] = [hf.make_opts(sun=sun, **opts) for sun in SUN_DAY]
        s["outs"] = [_outputs(cams, fields) for _ in SUN_DAY]
        return s
    s["outs"] = _outputs(cams, fields)
    if c["kind"] in ("render", "edit"):
        s["opts"] = hf.make_opts(**opts)
    elif c["kind"] == "march":
        s["opts"] = hf.make_march_opts(steps=c["steps"])
    elif c["kind"] == "scatter":
        s["opts"] = hf.make_scatter_opts(nu=c["nu"], nv=c["nv"], nz=c["nz"])
    elif c["kind"] in ("voxel", "bake"):
        s["grid"] = (c["vx"], c["vy"], c["vz"])
        s["opts"] = hf.make_voxel_opts(inner=c["inner"])
        if c["kind"] == "voxel":
            hf.hf_voxel_build(ctx, *s["grid"])
    elif c["kind"] == "serve":
        s["opts"] = opts["flags"]
        s["requests"], s["to"] = [], []
        for i, cam in enumerate(cams):
            s["requests"].append(dict(kind="render", arrival=0.0, cam=cam))
            s["to"].append(s["outs"][1][i])
            if i * 4 // len(cams) < (i + 1) * 4 // len(cams):
                s["requests"].append(dict(kind="edit", arrival=0.0, edit=edits[i * 4 // len(cams)]))
                s["to"].append(None)
        for x, y, b in reversed(edits):
            old = cells[y:y + b.shape[0], x:x + b.shape[1]].copy()
            s["requests"].append(dict(kind="edit", arrival=0.0, edit=(x, y, old)))
            s["to"].append(None)
    return s


def run(s):
    ctx, kind = s["world"].handle, s["kind"]
    if kind == "suns":
        for opts, (_, views) in zip(s["opts"], s["outs"]):
            hf.hf_render(ctx, s["cams"], views, opts)
        return [blocks for blocks, _ in s["outs"]]
    blocks, views = s["outs"]
    if kind == "edit":
        hf.hf_edit(ctx, *s["edits"][0])
    if kind in ("render", "edit"):
        hf.hf_render(ctx, s["cams"], views, s["opts"])
    elif kind == "march":
        hf.hf_render_march(ctx, s["cams"], views, s["opts"])
    elif kind == "scatter":
        hf.hf_render_scatter(ctx, s["cams"], views, None, s["opts"])
    elif kind == "serve":
        hf.hf_serve_replay(ctx, s["requests"], flags=s["opts"], outputs=s["to"])
    else:
        if kind == "bake":
            hf.hf_voxel_build(ctx, *s["grid"])
        hf.hf_render_voxel(ctx, s["cams"], views, s["opts"])
    return blocks


# -------------------------------------------------------- work and exactness

def _pixels(c):
    if c["pose"] == "mixed" or c["kind"] == "serve":
        total = 0
        for i in range(c["n"]):
            k = (1, 2, 3, 6)[i % 4] if c["kind"] == "serve" else \
                1 if 4 * i < c["n"] else 2 if 8 * i < 5 * c["n"] else 6
            total += max(1, c["w"] // k) * max(1, c["h"] // k)
        return total
    return c["n"] * c["w"] * c["h"]


def work(case):
    """Bytes: every output once, each pixel's cell once (at most the whole
    grid), edits, and what is built per pass.  Operations: about 60 per ray to
    make it, test one cell and shade it."""
    c = {**DEFAULTS, **case}
    px, cells = _pixels(c), c["W"] * c["H"]
    word = 2 if c["pairs"] else 4
    kind = c["kind"]
    out = 9 if kind in ("march", "voxel", "bake") else 15 if c["shadows"] else 14
    nbytes = px * out + min(word * cells, 4 * px)
    flops = 60 * px * (2 if c["shadows"] else 1)
    if "edit_w" in c:
        nbytes += 4 * c["edit_w"] * c["edit_h"] * (8 if kind == "serve" else 1)
    if kind == "suns":  # two images, and two sets of per-cell shadow bounds
        nbytes, flops = 2 * nbytes + 2 * 8 * cells, 2 * flops
    elif kind == "scatter":
        flops += 30 * c["n"] * c["nu"] * c["nv"] * c["nz"]
    elif kind == "bake":
        nbytes += 4 * cells + 256 * cells // (c["vx"] * c["vy"] * c["vz"]) // 7
    return {"bytes": nbytes, "flops": flops}


def _exact_depth(cells, cam):
    """Depth image of the flat cell-by-cell cast: exact 64-bit integer
    predicates in torch, the depth in float64."""
    W = cells.shape[1]
    H = cells.shape[0]
    grid = torch.from_numpy(cells.view(np.int32)).cuda().flatten().long()
    w, h = int(cam["w"]), int(cam["h"])
    pix = torch.arange(w * h, device="cuda")
    a, b = 2 * (pix % w) + 1 - w, h - 1 - 2 * (pix // w)
    o = [int(v) for v in cam["o"]]
    d = [int(cam["f"][k]) + a * int(cam["r"][k]) + b * int(cam["u"][k]) for k in range(3)]
    depth = torch.full((w * h,), math.inf, dtype=torch.float64, device="cuda")
    ad = [d[0].abs(), d[1].abs()]
    g = [torch.where(d[k] < 0, -1, 1) for k in range(2)]
    c = [torch.full_like(pix, o[k] >> 16) - ((d[k] < 0) & (o[k] % 65536 == 0)).long()
         for k in range(2)]
    tn, td = torch.zeros_like(pix), torch.ones_like(pix)
    length = sum(v.double() ** 2 for v in d).sqrt() / 65536
    dz = d[2]
    far = 1 << 40  # the exit of a ray that never leaves its column
    while pix.numel():
        inside = (c[0] >= 0) & (c[0] < W) & (c[1] >= 0) & (c[1] < H)
        word = grid[torch.where(inside, c[1] * W + c[0], 0)]
        f, m, t = word & 255, (word >> 8) & 255, (word >> 16) & 255
        slab = m > f
        num = [g[k] * (((c[k] + (g[k] > 0)) << 16) - o[k]) for k in range(2)]
        cmp = num[0] * ad[1] - num[1] * ad[0]
        xf = (ad[0] > 0) & ((ad[1] == 0) | (cmp <= 0))
        yf = (ad[1] > 0) & ((ad[0] == 0) | (cmp >= 0))
        en = torch.where(xf, num[0], torch.where(yf, num[1], far))
        ed = torch.where(xf, ad[0], torch.where(yf, ad[1], 1))

        def side(hgt, n_, d_):  # sign of z(n/d) - height
            return (o[2] - (hgt << 16)) * d_ + n_ * dz

        i0, i1, i2 = side(f, tn, td), side(m, tn, td), side(t, tn, td)
        e0, e1, e2 = side(f, en, ed), side(m, en, ed), side(t, en, ed)
        at_in = (i0 <= 0) | (slab & (i1 >= 0) & (i2 <= 0))
        to_top = slab & (dz < 0) & (i2 > 0) & (e2 <= 0)
        to_floor = (dz < 0) & (e0 <= 0)
        to_under = slab & (dz > 0) & (i1 < 0) & (e1 >= 0)
        hz = torch.where(to_top, t, torch.where(to_under, m, f))
        t_in = tn.double() / td.double()
        t_z = ((hz << 16) - o[2]).double() / torch.where(dz == 0, 1, dz).double()
        hit = inside & (at_in | to_top | to_floor | to_under)
        depth[pix[hit]] = (torch.where(at_in, t_in, t_z) * length)[hit]
        keep = (inside & ~hit).nonzero()[:, 0]
        c = [torch.where(xf, c[0] + g[0], c[0]), torch.where(yf, c[1] + g[1], c[1])]
        pix, tn, td, dz, length = pix[keep], en[keep], ed[keep], dz[keep], length[keep]
        c, ad, g = [v[keep] for v in c], [v[keep] for v in ad], [v[keep] for v in g]
    return depth


def exact(case, seed):
    """The depths of the exact cast, for up to a few million rays on a middling grid.  The
    comparison renderers (march, scatter, voxel) are defined as float32
    operations in a fixed order, so they have no value of higher precision."""
    c = {**DEFAULTS, **case}
    if c["kind"] not in ("render", "edit", "suns") or _pixels(c) > 3000000 or c["W"] + c["H"] > 6000:
        return None
    c, cells, cams, edits = _inputs(case, seed)
    if c["kind"] == "edit":
        x, y, b = edits[0]
        cells[y:y + b.shape[0], x:x + b.shape[1]] = b
    one = dict(hit_cell=None, layer=None, face=None, rgba=None, shadow=None,
               depth=torch.cat([_exact_depth(cells, k) for k in cams]))
    return [one, one] if c["kind"] == "suns" else one
