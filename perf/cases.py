"""What a user of this framework has it do, as cases that can be timed.

A case is one call of the matching path (pyramids, coarse-to-fine matching, final filter) on a
batch of image pairs, one pyramid build, or one sparse-to-dense interpolation, through the
package's public entry points.  Image pairs are made on the GPU from the seed: layered textured
polygons under rigid motions (as `synth.sintel_like_pair`), an expansion with gain and bias (as
`synth.kitti_like_pair`) or one affine motion (as `synth.noise_affine_pair`), with textures that
are smoothed noise, as those generators', or a 1/f mixture of octaves, as photographs are.
"""
import math

import torch

from paper_1704_03217_gb300 import api

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def _step(name, w, h, batch, form, content, **prm):
    c = {"kind": "step", "w": w, "h": h, "batch": batch, "form": form, "content": content,
         "levels": 5, "color": 1, "descriptor": 0, "seed_stride": 3, "patch_fwd": 15,
         "patch_bwd": 11, "iters_coarse": 4, "rs_grid": 0}
    c.update(prm)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small gray pair, each library call launched by itself: the least work that a
        # program hands over, where launches and the host's time count
        _step("gray_256x192", 256, 192, 1, "eager", "affine", levels=3, color=0, patch_fwd=8,
              patch_bwd=8, iters_coarse=6),
        # a camera's stream: one pair per frame, direction descriptor, replayed as a CUDA graph
        _step("live_gray_dir_640x480", 640, 480, 1, "graph", "natural", levels=4, color=0,
              descriptor=1),
        # one Sintel-shaped colour pair, as an interactive user runs it
        _step("pair_1024x436", 1024, 436, 1, "eager", "layers"),
        # the benchmark's step: 16 Sintel-shaped colour pairs resident on the GPU
        _step("batch16_1024x436", 1024, 436, 16, "graph", "layers"),
        # the same with the direction-only descriptor (bit-planes), and with the gray one
        _step("batch16_dir_1024x436", 1024, 436, 16, "graph", "layers", descriptor=1),
        _step("batch16_gray_1024x436", 1024, 436, 16, "graph", "layers", color=0),
        # driving sequences: a few KITTI-shaped pairs (odd height) a call
        _step("batch4_kitti_1242x375", 1242, 375, 4, "eager", "expansion"),
        # one full-HD pair of photograph-like frames
        _step("hd_natural_1920x1080", 1920, 1080, 1, "graph", "natural"),
        # one tick of a server: pairs of unequal sizes in shared launches
        {"name": "mixed_12", "kind": "mixed", "pairs": 12, "content": "layers", "levels": 5,
         "sizes": 0},
        # the paper's own setting, every pixel a seed, random search on the export grid only
        _step("dense_c3_1024x436", 1024, 436, 1, "graph", "layers", levels=3, seed_stride=1,
              rs_grid=3),
        # the pyramids of two full-HD frames of a sequence (each is kept and matched twice)
        {"name": "pyramid_1920x1080", "kind": "pyramid", "w": 1920, "h": 1080, "frames": 2,
         "levels": 5, "color": 1, "descriptor": 0, "content": "natural"},
        # a dense flow from one pair's exported matches
        {"name": "interp_1024x436", "kind": "interp", "w": 1024, "h": 436, "k": 16, "mode": 0,
         "content": "layers"},
    ]


# the sizes of a mixed batch: the benchmark's batched and served workloads', and odd ones
MIXED = [[(320, 240), (640, 480), (1024, 436), (1242, 375), (1920, 1080)],
         [(640, 480), (1280, 720), (1920, 1080), (1024, 436)],
         [(317, 241), (641, 359), (853, 481), (1025, 437)]]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["step", "dense", "mixed", "pyramid", "interp"], [6, 1, 1, 1, 1])[0]
    content = rng.choice(["layers", "natural", "expansion", "affine"])
    if kind == "mixed":
        return {"kind": "mixed", "pairs": rng.randint(2, 12), "content": content,
                "levels": rng.randint(4, 5), "sizes": rng.randrange(len(MIXED))}
    if kind == "pyramid":
        return {"kind": "pyramid", "w": _log_int(rng, 256, 1920), "h": _log_int(rng, 192, 1080),
                "frames": rng.randint(1, 2), "levels": rng.randint(3, 5),
                "color": rng.randint(0, 1), "descriptor": rng.randint(0, 1), "content": content}
    if kind == "interp":
        return {"kind": "interp", "w": _log_int(rng, 256, 1024), "h": _log_int(rng, 192, 436),
                "k": rng.choice([8, 16, 16]), "mode": rng.randint(0, 2), "content": content}
    if kind == "dense":
        return _step(None, _log_int(rng, 160, 1024), _log_int(rng, 120, 436), 1,
                     rng.choice(["eager", "graph"]), content, levels=3, seed_stride=1,
                     color=rng.randint(0, 1), rs_grid=3)
    w, h = _log_int(rng, 240, 1920), _log_int(rng, 180, 1080)
    most = max(1, min(16, 16 * 1024 * 436 // (w * h)))
    pf, pb = rng.choice([(15, 11), (15, 11), (11, 11), (8, 8)])
    return _step(None, w, h, _log_int(rng, 1, most), rng.choice(["eager", "graph"]), content,
                 levels=rng.randint(3 if w * h < 320 * 240 else 4, 5), color=rng.randint(0, 1),
                 descriptor=rng.randint(0, 1), seed_stride=rng.choice([2, 3, 3, 4]), patch_fwd=pf,
                 patch_bwd=pb, iters_coarse=rng.choice([4, 4, 6]))


def _params(case):
    keys = ("levels", "color", "descriptor", "seed_stride", "patch_fwd", "patch_bwd",
            "iters_coarse", "rs_grid")
    return api.Params(**{k: case[k] for k in keys if k in case})


# ------------------------------------------------------------------ image pairs
def _blur(x, sigma):
    """Gaussian of an (..., h, w) stack, borders reflected; plain shifted sums, so that the same
    seed gives the same bytes in every process."""
    r = max(1, int(math.ceil(3 * sigma)))
    wt = [math.exp(-0.5 * (i / sigma) ** 2) for i in range(-r, r + 1)]
    s = sum(wt)
    for d in (-1, -2):
        n = x.shape[d]
        i = torch.arange(-r, n + r, device=x.device).abs()
        i = torch.minimum(i, 2 * (n - 1) - i)
        p = x.index_select(d, i)
        x = sum((wt[k] / s) * p.narrow(d, k, n) for k in range(2 * r + 1))
    return x


def _texture(g, rng, h, w, ch, content):
    """(ch, h, w) float texture, 0..255."""
    if content == "natural":               # octaves of equal variance: a 1/f amplitude spectrum
        t = torch.zeros(ch, h, w, device=DEV)
        for o in range(6):
            hh, ww = max(8, h >> o), max(8, w >> o)
            n = _blur(torch.randn(ch, hh, ww, generator=g, device=DEV), 1.0)
            n = n / n.std()
            t = t + torch.nn.functional.interpolate(n[None], size=(h, w), mode="bilinear",
                                                    align_corners=False)[0]
        if ch == 3:                        # the channels of a photograph go together
            t = 0.8 * t[:1] + 0.2 * t
    else:
        t = _blur(torch.rand(ch, h, w, generator=g, device=DEV), rng.uniform(1.0, 2.5))
    z = (t - t.mean()) / t.std()
    return (127.5 + 49.5 * z).clamp(0, 255)


def _sample(img, x, y):
    h, w = img.shape[-2:]
    grid = torch.stack([2 * x / (w - 1) - 1, 2 * y / (h - 1) - 1], -1)
    return torch.nn.functional.grid_sample(img[None], grid[None], mode="bilinear",
                                           padding_mode="border", align_corners=True)[0]


def _pair(seed, w, h, ch, content):
    """Two uint8 images (h, w[, 3]) and the flow (2, h, w) between them."""
    import random
    rng = random.Random(seed)
    g = torch.Generator(device=DEV).manual_seed(seed)
    yy, xx = torch.meshgrid(torch.arange(h, device=DEV, dtype=torch.float32),
                            torch.arange(w, device=DEV, dtype=torch.float32), indexing="ij")
    cx, cy = (w - 1) / 2, (h - 1) / 2
    base = _texture(g, rng, h, w, ch, content)
    if content == "expansion":             # forward motion, then another exposure
        k = 200.0 / 1297 * rng.uniform(0.5, 1.0)
        f1, fx, fy = base, k * (xx - cx), k * (yy - cy)
        f2 = _sample(base, cx + (xx - cx) / (1 + k), cy + (yy - cy) / (1 + k))
        f2 = f2 * rng.uniform(0.8, 1.2) + rng.uniform(-20, 20)
    elif content == "affine":
        th, tx, ty = math.radians(rng.uniform(-3, 3)), rng.uniform(-12, 12), rng.uniform(-12, 12)
        c, s = math.cos(th), math.sin(th)
        qx, qy = xx - cx - tx, yy - cy - ty
        f1, f2 = base, _sample(base, c * qx + s * qy + cx, -s * qx + c * qy + cy)
        fx = c * (xx - cx) - s * (yy - cy) + cx + tx - xx
        fy = s * (xx - cx) + c * (yy - cy) + cy + ty - yy
    else:                                  # layers of polygons over a background
        bx, by = rng.uniform(-8, 8), rng.uniform(-8, 8)
        f1, f2 = base, _sample(base, xx - bx, yy - by)
        fx, fy = torch.full_like(xx, bx), torch.full_like(xx, by)
        tm = min(150.0, w / 8)
        for _ in range(rng.randint(3, 6)):
            tex = _texture(g, rng, h, w, ch, content)
            if ch == 3:
                sc = torch.tensor([rng.uniform(0.5, 1.0) for _ in range(3)], device=DEV)
                of = torch.tensor([rng.uniform(0, 80) for _ in range(3)], device=DEV)
                tex = (tex * sc[:, None, None] + of[:, None, None]).clamp(0, 255)
            r = rng.uniform(0.12, 0.3) * min(w, h)
            px, py = rng.uniform(r, w - r), rng.uniform(r, h - r)
            tx, ty = rng.uniform(-tm, tm), rng.uniform(-tm, tm)
            th, sc = math.radians(rng.uniform(-4, 4)), rng.uniform(0.93, 1.07)
            c, s = sc * math.cos(th), sc * math.sin(th)
            n = rng.randint(5, 8)
            ang = sorted(rng.uniform(0, 2 * math.pi) for _ in range(n))
            rad = [r * rng.uniform(0.75, 1.0) for _ in range(n)]

            def inside(x, y):
                m = torch.ones_like(x, dtype=torch.bool)
                for i in range(n):
                    x0, y0 = px + rad[i] * math.cos(ang[i]), py + rad[i] * math.sin(ang[i])
                    j = (i + 1) % n
                    x1, y1 = px + rad[j] * math.cos(ang[j]), py + rad[j] * math.sin(ang[j])
                    m &= ((x1 - x0) * (y - y0) - (y1 - y0) * (x - x0)) >= 0
                return m

            in1 = inside(xx, yy)
            f1 = torch.where(in1, tex, f1)
            fx = torch.where(in1, c * (xx - px) - s * (yy - py) + px + tx - xx, fx)
            fy = torch.where(in1, s * (xx - px) + c * (yy - py) + py + ty - yy, fy)
            det = c * c + s * s
            qx, qy = xx - px - tx, yy - py - ty
            ux, uy = (c * qx + s * qy) / det + px, (-s * qx + c * qy) / det + py
            f2 = torch.where(inside(ux, uy), _sample(tex, ux, uy), f2)
        p = torch.nn.functional.pad(f2[None], (1, 1, 0, 0), mode="replicate")[0]
        f2 = (p[..., :-2] + p[..., 1:-1] + p[..., 2:]) / 3           # mild motion blur
    out = []
    for f in (f1, f2):
        u = f.round().clamp(0, 255).to(torch.uint8)
        out.append(u[0].contiguous() if ch == 1 else u.permute(1, 2, 0).contiguous())
    return out[0], out[1], torch.stack([fx, fy])


# ------------------------------------------------------------------ preparation
def _prepare_step(case, seed):
    w, h, n = case["w"], case["h"], case["batch"]
    prm = _params(case)
    pairs = [_pair(1000 * seed + k, w, h, 3 if case["color"] else 1, case["content"])
             for k in range(n)]
    i1, i2 = [p[0] for p in pairs], [p[1] for p in pairs]
    m = api.PairMatcher(prm, w, h, batch=n)
    m.rows.zero_()                         # rows past a pair's count stay as they are here
    if case["form"] == "graph":
        m.capture(i1, i2)
    return {"case": case, "m": m, "i1": i1, "i2": i2, "fields": _fields(m.ws)}


def _prepare_mixed(case, seed):
    prm = _params(case)
    sizes = [MIXED[case["sizes"]][k % len(MIXED[case["sizes"]])] for k in range(case["pairs"])]
    pairs = [_pair(1000 * seed + k, w, h, 3, case["content"]) for k, (w, h) in enumerate(sizes)]
    st = {"case": case, "prm": prm, "i1": [p[0] for p in pairs], "i2": [p[1] for p in pairs]}
    st["p1"] = [api.Pyramid(prm, w, h) for w, h in sizes]
    st["p2"] = [api.Pyramid(prm, w, h) for w, h in sizes]
    st["ws"] = [api.Workspace(prm, w, h, w, h) for w, h in sizes]
    st["rows"], st["count"] = [], []
    for ws in st["ws"]:
        nx, ny, *_ = ws.layout(0, 0)
        st["rows"].append(torch.zeros(nx * ny, 4, dtype=torch.int32, device=DEV))
        st["count"].append(torch.zeros(1, dtype=torch.int32, device=DEV))
    st["fields"] = _fields(st["ws"])
    return st


def _fields(wss):
    """The level-0 fields of every workspace as views: displacements of both directions, and for
    a few pairs the costs and flags too."""
    out = []
    for ws in wss:
        for d in (0, 1):
            nx, ny, ou, oc, of = ws.layout(0, d)
            n = nx * ny
            f = {"u": ws.buf[ou:ou + 4 * n].view(torch.int16).view(ny, nx, 2)}
            if len(wss) <= 4:
                f["cost"] = ws.buf[oc:oc + 8 * n].view(torch.int64).view(ny, nx)
                f["flags"] = ws.buf[of:of + n].view(ny, nx)
            out.append(f)
    return out


def _prepare_pyramid(case, seed):
    w, h, ch = case["w"], case["h"], 3 if case["color"] else 1
    prm = _params(case)
    a, b, _ = _pair(1000 * seed, w, h, ch, case["content"])
    imgs = [a, b][:case["frames"]]
    pyrs = [api.Pyramid(prm, w, h) for _ in imgs]
    out = [{"desc": [p.desc_padded(s, l) for s in range(1 + case["color"])
                     for l in range(case["levels"])],
            "image": [p.cimage(s, l) for s in range(1 + case["color"])
                      for l in range(case["levels"])]} for p in pyrs]
    return {"case": case, "prm": prm, "imgs": imgs, "pyrs": pyrs, "out": out}


def _interp_inputs(case, seed):
    """An image and the matches of its grid-3 seeds: the flow, in whole pixels, where the pair
    can be matched (about three fifths of the seeds; the gaps are connected patches, as
    occlusions and removed regions are)."""
    w, h = case["w"], case["h"]
    img, _, flow = _pair(1000 * seed, w, h, 3, case["content"])
    g = torch.Generator(device=DEV).manual_seed(seed + 7)
    gap = _blur(torch.randn(h, w, generator=g, device=DEV), 8.0)
    gap = gap / gap.std()
    y, x = torch.meshgrid(torch.arange(1, h, 3, device=DEV), torch.arange(1, w, 3, device=DEV),
                          indexing="ij")
    keep = (gap[y, x] < 0.5) & (torch.rand(y.shape, generator=g, device=DEV) < 0.9)
    x, y = x[keep], y[keep]
    u = flow[:, y, x].round().int()
    rows = torch.stack([x.int(), y.int(), x.int() + u[0], y.int() + u[1]], -1).contiguous()
    return img, rows


def _prepare_interp(case, seed):
    img, rows = _interp_inputs(case, seed)
    prm = api.Params(levels=3)
    ip = api.InterpParams(k=case["k"], mode=case["mode"])
    pyr = api.build_pyramid(prm, img)
    cnt = torch.tensor([rows.shape[0]], dtype=torch.int32, device=DEV)
    _, ws = api.interpolate(prm, pyr, rows, cnt, ip)
    return {"case": case, "prm": prm, "pyr": pyr, "rows": rows, "count": cnt, "ip": ip, "ws": ws}


def prepare(case, seed):
    return {"step": _prepare_step, "mixed": _prepare_mixed, "pyramid": _prepare_pyramid,
            "interp": _prepare_interp}[case["kind"]](case, seed)


# ------------------------------------------------------------------ one pass
def run(state):
    c = state["case"]
    if c["kind"] == "step":
        m = state["m"]
        if c["form"] == "graph":
            m.replay()
        else:
            m.enqueue(state["i1"], state["i2"])
        return {"rows": m.rows, "count": m.count, "fields": state["fields"]}
    if c["kind"] == "mixed":
        prm, n = state["prm"], len(state["ws"])
        api.build_pyramids(prm, state["i1"] + state["i2"], state["p1"] + state["p2"])
        api.match_batch(prm, state["p1"], state["p2"], list(range(n)), state["ws"])
        api.filter_batch(prm, state["ws"], state["rows"], state["count"])
        return {"rows": state["rows"], "count": state["count"], "fields": state["fields"]}
    if c["kind"] == "pyramid":
        api.build_pyramids(state["prm"], state["imgs"], state["pyrs"])
        return state["out"]
    flow, _ = api.interpolate(state["prm"], state["pyr"], state["rows"], state["count"],
                              state["ip"], state["ws"])
    return flow


# ------------------------------------------------------------------ the work it needs
def _pyramid_px(w, h, levels):
    n = 0
    for _ in range(levels):
        n, w, h = n + w * h, (w + 1) // 2, (h + 1) // 2
    return n


def _step_work(prm, w, h):
    """One pair: the images in, every descriptor written and read once, the matches out; and the
    multiply-adds of Eq. 3 for every candidate that the method names (the exhaustive
    initialisation's among them)."""
    ch = 3 if prm.color else 1
    one = 2 if prm.descriptor else 16                            # bits of a descriptor value
    px = _pyramid_px(w, h, prm.levels)
    s = prm.seed_stride
    seeds = (w // s) * (h // s)
    by = 2 * w * h * ch + 2 * (1 + prm.color) * px * 2 * ch * one / 8 * 2 + 16 * seeds
    cw, chh = -(-w >> (prm.levels - 1)), -(-h >> (prm.levels - 1))
    mac = 2 * ch * (prm.patch_fwd ** 2 + prm.patch_bwd ** 2) / 2
    ev = api.nominal_evals(prm, w, h, w, h) + 2 * (cw // s) * (chh // s) * cw * chh
    return by, 2 * ev * mac


def work(case):
    prm = _params(case)
    if case["kind"] == "step":
        by, fl = _step_work(prm, case["w"], case["h"])
        return {"bytes": by * case["batch"], "flops": fl * case["batch"]}
    if case["kind"] == "mixed":
        by = fl = 0
        for k in range(case["pairs"]):
            b, f = _step_work(prm, *MIXED[case["sizes"]][k % len(MIXED[case["sizes"]])])
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    if case["kind"] == "pyramid":
        ch = 3 if case["color"] else 1
        px = _pyramid_px(case["w"], case["h"], case["levels"])
        out = (1 + case["color"]) * px * (4 * ch + ch)            # int16 gradients, converted bytes
        return {"bytes": case["frames"] * (case["w"] * case["h"] * ch + out),
                "flops": case["frames"] * (1 + case["color"]) * px * ch * 40}
    n = case["w"] * case["h"]
    # the descriptor in, the neighbour lists and the flow out; a step's sums and comparisons for
    # every neighbour's entry once, and a weighted affine fit per pixel
    return {"bytes": n * (12 + 8 * case["k"] + 8), "flops": n * case["k"] * (4 * 2 + 40)}


# ------------------------------------------------------------------ in 64 bits
def _knn(cost, rows, h, w, k):
    """(h w, k) keys d << 32 | index of the k geodesically nearest matches, by relaxation."""
    n, big = h * w, (1 << 62)
    key = torch.full((n + 1, k), big, dtype=torch.int64, device=DEV)      # row n: outside
    p = rows[:, 1].long() * w + rows[:, 0].long()
    first = torch.full((n,), big, dtype=torch.int64, device=DEV)
    idx = torch.arange(rows.shape[0], device=DEV)
    first.scatter_reduce_(0, p, idx, "amin")
    key[:n, 0] = first
    x, y = torch.arange(n, device=DEV) % w, torch.arange(n, device=DEV) // w
    nb = torch.stack([torch.where(x > 0, torch.arange(n, device=DEV) - 1, n),
                      torch.where(x < w - 1, torch.arange(n, device=DEV) + 1, n),
                      torch.where(y > 0, torch.arange(n, device=DEV) - w, n),
                      torch.where(y < h - 1, torch.arange(n, device=DEV) + w, n)], 1)
    cst = torch.cat([cost.reshape(-1), cost.new_zeros(1)])
    live = torch.arange(n, device=DEV)
    low = (1 << 32) - 1
    while live.numel():
        moved = []
        for part in live.split(1 << 18):
            q = nb[part]
            cand = key[q] + ((cst[part][:, None] + cst[q]) << 32)[..., None]
            c = torch.cat([key[part], cand.reshape(part.numel(), 4 * k)], 1)
            c = torch.where(c >= big, big, c)
            by = torch.where(c >= big, c, ((c & low) << 31) | (c >> 32)).sort(1)[0]
            lab = by >> 31
            dup = torch.zeros_like(by, dtype=torch.bool)
            dup[:, 1:] = lab[:, 1:] == lab[:, :-1]
            back = ((by & ((1 << 31) - 1)) << 32) | (by >> 31)
            new = torch.where(dup | (by >= big), big, back).sort(1)[0][:, :k]
            ch = (new != key[part]).any(1)
            moved.append((part[ch], new[ch]))
        for part, new in moved:
            key[part] = new
        ch = torch.cat([m[0] for m in moved])
        if ch.numel() == 0:
            break
        mark = torch.zeros(n + 1, dtype=torch.bool, device=DEV)
        mark[nb[ch].reshape(-1)] = True
        live = mark[:n].nonzero()[:, 0]
    return key[:n], big


def exact(case, seed):
    """The interpolation's flow in 64 bits (the other outputs are whole numbers)."""
    if case["kind"] != "interp":
        return None
    img, rows = _interp_inputs(case, seed)
    h, w, k = case["h"], case["w"], case["k"]
    v = img.permute(2, 0, 1).long()
    yy = torch.arange(-2, h + 2, device=DEV).clamp(0, h - 1)
    xx = torch.arange(-2, w + 2, device=DEV).clamp(0, w - 1)
    v = v[:, yy][:, :, xx]
    d, s = (-1, -2, 0, 2, 1), (1, 4, 6, 4, 1)
    tot = torch.zeros(h, w, dtype=torch.int64, device=DEV)
    for a, b in ((d, s), (s, d)):          # Sobel of side 5 along x, then along y
        row = sum(a[i] * v[:, :, i:i + w] for i in range(5))
        tot += sum(b[j] * row[:, j:j + h] for j in range(5)).abs().sum(0)
    key, big = _knn(1 + (tot >> 10), rows, h, w, k)
    ok = key < big
    dist = (key >> 32).double()
    i = torch.where(ok, key & ((1 << 32) - 1), 0)
    wt = torch.where(ok, torch.exp(-(dist - dist[:, :1]) / 32.0), torch.zeros_like(dist))
    r = rows.double()[i]
    px = torch.arange(h * w, device=DEV) % w
    py = torch.arange(h * w, device=DEV) // w
    f = r[..., 2:] - r[..., :2]
    sw = wt.sum(1)
    nw = (wt[..., None] * f).sum(1) / sw.clamp(min=1e-300)[:, None]
    la = case["mode"] == 2 or (case["mode"] == 0 and rows.shape[0] * 10000 > 220 * w * h)
    if la:
        q = torch.stack([r[..., 0] - px[:, None], r[..., 1] - py[:, None],
                         torch.ones_like(wt)], -1)
        M = torch.einsum("ne,nea,neb->nab", wt, q, q)
        b = torch.einsum("ne,nea,nef->naf", wt, q, f)

        def det3(m):
            return (m[:, 0, 0] * (m[:, 1, 1] * m[:, 2, 2] - m[:, 1, 2] * m[:, 2, 1])
                    - m[:, 0, 1] * (m[:, 1, 0] * m[:, 2, 2] - m[:, 1, 2] * m[:, 2, 0])
                    + m[:, 0, 2] * (m[:, 1, 0] * m[:, 2, 1] - m[:, 1, 1] * m[:, 2, 0]))

        det = det3(M)
        good = det > 1e-6 * sw ** 3
        c = []
        for j in range(2):                 # Cramer's rule for the constant term
            Mj = M.clone()
            Mj[:, :, 2] = b[:, :, j]
            c.append(det3(Mj) / torch.where(good, det, torch.ones_like(det)))
        nw = torch.where(good[:, None], torch.stack(c, 1), nw)
    return torch.where((sw > 0)[:, None], nw, torch.zeros_like(nw)).view(h, w, 2)
