"""The measured cases of the framework: the calls a program makes, over the
sizes it makes them at.

Tiles are H&E-like (background, stroma discs, nuclei singly, overlapping, in
clusters or in chains, optional red blood cells and ramp corridors, noise,
blur) and are painted on the GPU from the seed alone.  Sizes and densities are
those of the workloads this repository is tested and benchmarked on: the 512 x
512 tile with 60 nuclei, the 4096 x 4096 tile with 3000, the mixed batch with
sides 1024 to 4096 and 0 to 5000 nuclei per 4096 x 4096, the worst-case tile
with 8000 nuclei, half of them in long chains, and ramp corridors.
"""
import math

import numpy as np
import torch

import paper_1209_3332_gb300 as P

FULL = 4096 * 4096  # pixels of the tile that densities are quoted for

_pipes = {}


def _pipe():
    """The handle a program keeps for its lifetime (default parameters)."""
    dev = torch.cuda.current_device()
    if dev not in _pipes:
        _pipes[dev] = P.Pipe(dev)
    return _pipes[dev]


# ---- cases -----------------------------------------------------------------


def listed():
    return [
        # a thumbnail or a region of interest, one call at a time: launches and latency
        dict(name="plain_512", kind="plain", W=512, H=512, nuclei=3840, stroma=0),
        # a tile at the ragged edge of a slide, odd in both sides: no wide access fits its rows
        dict(name="plain_1025x2049", kind="plain", W=1025, H=2049, nuclei=3000, stroma=150),
        # the paper's 4K x 4K tile, one call per tile, features after the count is known
        dict(name="plain_4096", kind="plain", W=4096, H=4096, nuclei=3000, stroma=150),
        # a batch as a slide's tiler hands it over: sides 1024 to 4096, empty to dense
        dict(name="batch_mixed_12", kind="batch", n=12, W=0, H=0, nuclei=0, stroma=0),
        # the throughput form on the benchmark tile: 16 tiles of 4K x 4K
        dict(name="batch_16x4096", kind="batch", n=16, W=4096, H=4096, nuclei=3000, stroma=150),
        # worst-case tissue: long chains of touching nuclei and faint ramps that fronts travel along
        dict(name="batch_chains_4x4096", kind="batch", n=4, W=4096, H=4096, nuclei=8000, stroma=0, chains=True),
        # a server: tiles in pinned host memory, four groups of four, two groups in flight
        dict(name="served_16x2048", kind="served", n=16, group=4, W=2048, H=2048, nuclei=3000, stroma=150),
        # splitting the touching objects of one small tile
        dict(name="watershed_1024", kind="watershed", n=1, W=1024, H=1024, nuclei=3000, stroma=150, h=1),
        # and of a batch of benchmark tiles
        dict(name="watershed_8x4096", kind="watershed", n=8, W=4096, H=4096, nuclei=3000, stroma=150, h=1),
        # edges of the hematoxylin planes of a batch, and the edge count of every object
        dict(name="canny_8x4096", kind="canny", n=8, W=4096, H=4096, nuclei=3000, stroma=150, radius=3),
        # the opening by the paper's 19 x 19 disk of one hematoxylin plane
        dict(name="morph_open_4096", kind="morph", W=4096, H=4096, nuclei=3000, stroma=150, radius=9),
        # red blood cell mask of one tile
        dict(name="rbc_4096", kind="rbc", W=4096, H=4096, nuclei=3000, stroma=150, rbc=800),
    ]


def draw(rng):
    """One more case: any kind of call, sides spread over 256 to 4096, odd ones among them."""

    def side():
        return int(round(math.exp(rng.uniform(math.log(256), math.log(4096)))))

    kind = rng.choice(["plain", "plain", "batch", "batch", "served", "watershed", "canny", "morph", "rbc"])
    c = dict(kind=kind, W=side(), H=side(), nuclei=rng.randint(0, 5000), stroma=rng.randint(0, 250))
    if rng.random() < 0.2:
        c.update(chains=True, nuclei=8000, stroma=0)
    most = 4 if c.get("chains") else 16
    n = int(round(math.exp(rng.uniform(0, math.log(most)))))
    if kind == "batch":
        c["n"] = n
    elif kind == "served":
        c["n"], c["group"] = n, rng.randint(1, n)
    elif kind == "watershed":
        c["n"], c["h"] = min(n, 8), rng.choice([0, 1, 1, 2])
    elif kind == "canny":
        c["n"], c["radius"] = min(n, 8), rng.choice([0, 2, 3, 3, 4])
    elif kind == "morph":
        c["radius"] = rng.choice([3, 5, 9, 9, 9, 12, 15])
    elif kind == "rbc":
        c["rbc"] = rng.randint(0, 3000)
    return c


def _tiles(case):
    """(W, H, nuclei per 4096 x 4096, stroma per 4096 x 4096) of each tile."""
    n = case.get("n", 1)
    if case["W"]:
        return [(case["W"], case["H"], case["nuclei"], case["stroma"])] * n
    # the mixed batch: sides and densities spread evenly, the first tile empty
    out = []
    for i in range(n):
        side = (1024, 2048, 3072, 4096, 1536, 1000)[i % 6]
        out.append((side, side if i % 3 else side - 24 * (i % 4), 5000 * i // max(n - 1, 1), 250 * i // max(n - 1, 1)))
    return out


def work(case):
    px = sum(W * H for W, H, _, _ in _tiles(case))
    obj = sum(W * H * d / FULL for W, H, d, _ in _tiles(case)) * P.NFEAT * 4
    per_px = {
        "plain": 12,      # RGB in; hem8, labels and distance transform out
        "batch": 12,
        "served": 3,      # RGB over the host link; feature rows back
        "watershed": 12,  # labels and distance transform in, basins out
        "canny": 6,       # hem8 and labels in, edges out
        "morph": 2,
        "rbc": 4,
    }[case["kind"]]
    return {"bytes": per_px * px + (obj if case["kind"] in ("plain", "batch", "served") else 0), "flops": 0}


# ---- inputs -----------------------------------------------------------------

_BG, _NUC, _STROMA, _RBC = (225, 215, 228), (90, 60, 140), (200, 150, 190), (200, 60, 70)
_RAMP_END = (160, 110, 170)


def _paint(plane, W, H, cx, cy, a, b, th, first, step=512):
    """Ellipses into the index plane; a later one covers an earlier one."""
    if len(cx) == 0:
        return
    dev = plane.device
    r = int(math.ceil(max(a.max(), b.max()))) + 1
    oy, ox = torch.meshgrid(torch.arange(-r, r + 1, device=dev), torch.arange(-r, r + 1, device=dev), indexing="ij")
    step = max(1, min(step, (1 << 24) // ox.numel()))
    for i in range(0, len(cx), step):
        q = [torch.from_numpy(np.ascontiguousarray(v[i:i + step])).to(dev)[:, None, None] for v in (cx, cy, a, b, th)]
        x, y = torch.floor(q[0]) + ox, torch.floor(q[1]) + oy
        dx, dy = x - q[0], y - q[1]
        u, v = dx * torch.cos(q[4]) + dy * torch.sin(q[4]), -dx * torch.sin(q[4]) + dy * torch.cos(q[4])
        inside = (u * u / (q[2] * q[2]) + v * v / (q[3] * q[3]) <= 1) & (x >= 0) & (x < W) & (y >= 0) & (y < H)
        ids = torch.arange(first + i, first + i + x.shape[0], device=dev, dtype=torch.int32)[:, None, None].expand_as(inside)
        at = (y * W + x)[inside].long()
        plane.scatter_reduce_(0, at, ids[inside], "amax")


def _rgb(W, H, density, stroma_density, seed, chains=False, rbc=0):
    """One (H, W, 3) uint8 tile on the GPU."""
    r = np.random.default_rng(seed)
    n, ns = int(round(density * W * H / FULL)), int(round(stroma_density * W * H / FULL))
    nr = int(round(rbc * W * H / FULL))
    cols = [np.array([_BG], np.float32)]
    plane = torch.zeros(W * H, dtype=torch.int32, device="cuda")
    first = 1
    rad = r.uniform(40, 120, ns)
    _paint(plane, W, H, r.uniform(0, W, ns), r.uniform(0, H, ns), rad, rad, np.zeros(ns), first)
    cols.append(np.array(_STROMA) + r.integers(-5, 6, (ns, 3)))
    first += ns
    # nuclei: chains of 10 to 30 (half of them, on a worst-case tile), clusters of 2 to 6, singles
    a, b, th = r.uniform(4, 12, n), r.uniform(4, 12, n), r.uniform(0, math.pi, n)
    cx, cy, phi, turn = r.uniform(0, W, n), r.uniform(0, H, n), r.uniform(0, 2 * math.pi, n), r.uniform(-0.5, 0.5, n)
    kind, i = r.random(n), 0
    while i < n:
        u = kind[i]
        size = int(r.integers(10, 31)) if chains and u < 0.5 / 10 else int(r.integers(2, 7)) if u < (0.05 if chains else 0.06) + 0.06 else 1
        p = phi[i]
        for k in range(i + 1, min(i + size, n)):
            p = p + turn[k] if size > 6 else phi[k]
            d = (0.85 if size > 6 else 0.9) * 0.5 * (a[k - 1] + b[k - 1] + a[k] + b[k])
            cx[k], cy[k] = cx[k - 1] + d * math.cos(p), cy[k - 1] + d * math.sin(p)
        i += size
    _paint(plane, W, H, cx, cy, a, b, th, first)
    cols.append(np.array(_NUC) + r.integers(-8, 9, (n, 3)))
    first += n
    rad = r.uniform(3.5, 5.5, nr)
    _paint(plane, W, H, r.uniform(0, W, nr), r.uniform(0, H, nr), rad, rad, np.zeros(nr), first)
    cols.append(np.array(_RBC) + r.integers(-8, 9, (nr, 3)))
    first += nr
    if chains and W >= 512:
        # ramp corridors: bands of 9 rows over a cleared strip, their colour rising along the row
        for y in range(128, H - 128, 256):
            plane.view(H, W)[y - 14:y + 15, 128:W - 128] = 0
            at = torch.arange(W - 256, device="cuda", dtype=torch.int32)
            plane.view(H, W)[y - 4:y + 5, 128:W - 128] = first + (at if (y // 256) % 2 == 0 else at.flip(0))
        t = np.linspace(0, 1, W - 256)[:, None]
        cols.append(np.array(_STROMA) + (np.array(_RAMP_END) - np.array(_STROMA)) * t)
    table = torch.from_numpy(np.concatenate(cols).astype(np.float32)).cuda()
    g = torch.Generator(device="cuda")
    g.manual_seed(int(r.integers(1 << 40)))
    img = table[plane.view(H, W).long()]
    img += torch.randn(img.shape, generator=g, device="cuda") * 6.0
    w = [math.exp(-k * k / 2.0) for k in range(-3, 4)]
    for axis, size in ((0, H), (1, W)):
        out = torch.zeros_like(img)
        at = torch.arange(size, device="cuda")
        for k in range(-3, 4):
            out += img.index_select(axis, (at + k).clamp(0, size - 1)) * (w[k + 3] / sum(w))
        img = out
    return img.round_().clamp_(0, 255).to(torch.uint8)


def _images(case, seed):
    return [_rgb(W, H, d, s, (seed, i), bool(case.get("chains")), case.get("rbc", 0))
            for i, (W, H, d, s) in enumerate(_tiles(case))]


def _flat(sizes, dtype, per=1):
    """One zeroed buffer for all tiles of a batch, each at a 256-byte boundary, and the tiles' views."""
    unit = 256 // torch.empty(0, dtype=dtype).element_size()
    at, total = [], 0
    for W, H in sizes:
        at.append(total)
        total += -(-W * H * per // unit) * unit
    buf = torch.zeros(total, dtype=dtype, device="cuda")
    return buf, [buf[o:o + W * H * per].view(H, W) if per == 1 else buf[o:o + W * H * per] for o, (W, H) in zip(at, sizes)]


def _rows(W, H):
    """Feature rows a program has room for: twice the densest tile's objects."""
    return 64 + W * H // 800


def _batch(rgb):
    """Output buffers of a batch, and the argument list of seg_features_batch."""
    sizes = [(t.shape[1], t.shape[0]) for t in rgb]
    hem8, labels, edt = _flat(sizes, torch.uint8), _flat(sizes, torch.int32), _flat(sizes, torch.int32)
    nobj = torch.zeros(len(rgb), dtype=torch.int32, device="cuda")
    caps = [_rows(W, H) for W, H in sizes]
    feats = torch.zeros((sum(caps), P.NFEAT), dtype=torch.float32, device="cuda")
    tiles, at = [], 0
    for i, t in enumerate(rgb):
        tiles.append(dict(rgb=t, hem8=hem8[1][i], labels=labels[1][i], edt=edt[1][i], n_objects=nobj[i:i + 1],
                          feats=feats[at:at + caps[i]]))
        at += caps[i]
    return tiles, dict(hem8=hem8[0], labels=labels[0], edt=edt[0], n_objects=nobj, feats=feats)


def _segmented(case, seed):
    """The planes that the later operations take: hem8, labels, distance transform and object counts."""
    rgb = _images(case, seed)
    tiles, _ = _batch(rgb)
    for t in tiles:
        _pipe().seg_tile(t["rgb"], t["hem8"], t["labels"], t["edt"], t["n_objects"])
    counts = torch.cat([t["n_objects"] for t in tiles]).tolist()
    return tiles, counts


def prepare(case, seed):
    kind, pipe = case["kind"], _pipe()
    s = dict(kind=kind, pipe=pipe, case=case)
    if kind in ("plain", "batch"):
        s["tiles"], s["out"] = _batch(_images(case, seed))
    elif kind == "served":
        s["host"] = [t.cpu().pin_memory() for t in _images(case, seed)]
        s["feats"] = np.zeros((case["n"], _rows(case["W"], case["H"]), P.NFEAT), np.float32)  # the program's own table
    elif kind == "rbc":
        s["rgb"] = _images(case, seed)[0]
        s["out"] = torch.empty(s["rgb"].shape[:2], dtype=torch.uint8, device="cuda")
    elif kind == "morph":
        s["src"] = _segmented(case, seed)[0][0]["hem8"].clone()
        s["out"] = torch.empty_like(s["src"])
    elif kind == "watershed":
        tiles, counts = _segmented(case, seed)
        out = _flat([(t["labels"].shape[1], t["labels"].shape[0]) for t in tiles], torch.int32)
        nb = torch.zeros(len(tiles), dtype=torch.int32, device="cuda")
        s["tiles"] = [dict(labels=t["labels"], edt=t["edt"], n_objects=k, out=out[1][i], n_basins=nb[i:i + 1])
                      for i, (t, k) in enumerate(zip(tiles, counts))]
        s["out"] = dict(basins=out[0], n_basins=nb)
    elif kind == "canny":
        tiles, counts = _segmented(case, seed)
        edges = _flat([(t["hem8"].shape[1], t["hem8"].shape[0]) for t in tiles], torch.uint8)
        cnt = torch.zeros((len(tiles), max(t["feats"].shape[0] for t in tiles)), dtype=torch.int32, device="cuda")
        s["tiles"] = [dict(img=t["hem8"], labels=t["labels"], n_objects=k, edges=edges[1][i], counts=cnt[i, :k])
                      for i, (t, k) in enumerate(zip(tiles, counts))]
        s["out"] = dict(edges=edges[0], counts=cnt)
    return s


# ---- one pass ---------------------------------------------------------------


def run(s):
    pipe, kind, case = s["pipe"], s["kind"], s["case"]
    if kind == "plain":
        t = s["tiles"][0]
        pipe.seg_tile(t["rgb"], t["hem8"], t["labels"], t["edt"], t["n_objects"])
        k = int(t["n_objects"].item())  # the caller needs the count to ask for the features
        pipe.features_tile(t["hem8"], t["labels"], k, t["feats"])
        return s["out"]
    if kind == "batch":
        pipe.seg_features_batch(s["tiles"])
        return s["out"]
    if kind == "served":
        host, group = s["host"], case["group"]
        todo = [host[i:i + group] for i in range(0, len(host), group)]
        flying, res = [], []
        while todo or flying:
            if todo and len(flying) < 2:
                ticket = pipe.submit(todo[0])
                if ticket is not None:
                    flying.append(ticket)
                    todo.pop(0)
            if flying:
                got = pipe.poll(flying[0])
                if got is not None:
                    res += got
                    flying.pop(0)
        for i, r in enumerate(res):
            s["feats"][i, :r["feats"].shape[0]] = r["feats"]
        return dict(n_objects=np.array([r["n_objects"] for r in res], np.int32),
                    status=np.array([r["status"] for r in res], np.int32), feats=s["feats"])
    if kind == "watershed":
        if len(s["tiles"]) == 1:
            t = s["tiles"][0]
            pipe.watershed(t["labels"], t["edt"], t["n_objects"], t["out"], t["n_basins"], h=case["h"])
        else:
            pipe.watershed_batch(s["tiles"], h=case["h"])
        return s["out"]
    if kind == "canny":
        if len(s["tiles"]) == 1:
            t = s["tiles"][0]
            pipe.canny(t["img"], t["edges"], labels=t["labels"], n_objects=t["n_objects"], counts=t["counts"],
                       radius=case["radius"])
        else:
            pipe.canny_batch(s["tiles"], radius=case["radius"])
        return s["out"]
    if kind == "morph":
        pipe.morph_open(s["src"], s["out"], radius=case["radius"])
        return s["out"]
    pipe.rbc(s["rgb"], s["out"])
    return s["out"]


# ---- the same numbers in plain torch ---------------------------------------------


def _neighbours(x, fill, conn=8):
    """The shifted copies of a plane, `fill` beyond its border."""
    H, W = x.shape
    p = torch.nn.functional.pad(x[None, None], (1, 1, 1, 1), value=fill)[0, 0]
    return [p[1 + dy:1 + dy + H, 1 + dx:1 + dx + W] for dy in (-1, 0, 1) for dx in (-1, 0, 1)
            if (dy or dx) and (conn == 8 or not (dy and dx))]


def _settle(step, x):
    """step() until it changes nothing."""
    while True:
        y = x
        for _ in range(32):
            y = step(y)
        if torch.equal(x, y):
            return x
        x = y


def _exact_hem8(rgb):
    lut = np.array([math.floor(-math.log((v + 1) / 256.0) * 256.0 + 0.5) for v in range(256)])
    hs, es = np.array([0.650, 0.704, 0.286]), np.array([0.072, 0.990, 0.105])
    hs, es = hs / np.linalg.norm(hs), es / np.linalg.norm(es)
    rs = np.cross(hs, es)
    w = np.linalg.inv(np.stack([hs, es, rs / np.linalg.norm(rs)]))[:, 0]
    q = [int(round(100 * v * 2048)) for v in w]
    od = torch.from_numpy(lut).cuda()[rgb.long()]
    acc = sum(q[c] * od[..., c] for c in range(3))
    return ((acc + (1 << 18)) >> 19).clamp(0, 255)


def _exact_labels(hem, h=20, thr=10, amin=20, amax=1500):
    H, W = hem.shape
    m = hem.to(torch.uint8)

    def dilate(r):
        p = torch.nn.functional.pad(r[None, None], (1, 1, 1, 1))[0, 0]
        p = torch.maximum(torch.maximum(p[:-2], p[1:-1]), p[2:])
        return torch.minimum(torch.maximum(torch.maximum(p[:, :-2], p[:, 1:-1]), p[:, 2:]), m)

    r = _settle(dilate, (hem - h).clamp(min=0).to(torch.uint8))
    bg = hem - r.long() < thr
    seed = bg.clone()
    seed[1:-1, 1:-1] = False

    def flood(x):
        a, b, c, d = _neighbours(x, False, 4)
        return (x | a | b | c | d) & bg

    filled = ~_settle(flood, seed)
    big = H * W
    index = torch.arange(H * W, device="cuda", dtype=torch.int32).view(H, W)
    none = torch.full_like(index, big)

    def least(x):
        p = torch.nn.functional.pad(x[None, None], (1, 1, 1, 1), value=big)[0, 0]
        p = torch.minimum(torch.minimum(p[:-2], p[1:-1]), p[2:])
        return torch.where(filled, torch.minimum(torch.minimum(p[:, :-2], p[:, 1:-1]), p[:, 2:]), none)

    comp = _settle(least, torch.where(filled, index, none))
    roots, inverse, area = torch.unique(comp[filled], return_inverse=True, return_counts=True)
    keep = (area >= amin) & (area <= amax)
    number = torch.where(keep, torch.cumsum(keep.int(), 0), torch.zeros_like(area))
    labels = torch.zeros(H, W, dtype=torch.int64, device="cuda")
    labels[filled] = number[inverse]
    return labels, int(keep.sum())


def _exact_features(hem, labels, K):
    H, W = hem.shape
    f = torch.zeros(K, P.NFEAT, dtype=torch.float64, device="cuda")
    if K == 0:
        return f
    ys, xs = torch.nonzero(labels, as_tuple=True)
    obj, v = labels[ys, xs] - 1, hem[ys, xs]

    def total(x):
        return torch.zeros(K, dtype=torch.float64, device="cuda").index_add_(0, obj, x.double())

    def extreme(x, how):
        return torch.zeros(K, dtype=torch.float64, device="cuda").scatter_reduce_(0, obj, x.double(), how, include_self=False)

    def at(plane, dy, dx):
        return plane[(ys + dy).clamp(0, H - 1), (xs + dx).clamp(0, W - 1)]

    def same(dy, dx):
        inside = (ys + dy >= 0) & (ys + dy < H) & (xs + dx >= 0) & (xs + dx < W)
        return inside & (at(labels, dy, dx) == obj + 1)

    n = total(torch.ones_like(v))
    f[:, 0] = n
    f[:, 1] = total(sum((~same(dy, dx)).long() for dy, dx in ((-1, 0), (1, 0), (0, -1), (0, 1))))
    p = {(dy, dx): at(hem, dy, dx) for dy in (-1, 0, 1) for dx in (-1, 0, 1)}
    gx = p[-1, 1] + 2 * p[0, 1] + p[1, 1] - p[-1, -1] - 2 * p[0, -1] - p[1, -1]
    gy = p[1, -1] + 2 * p[1, 0] + p[1, 1] - p[-1, -1] - 2 * p[-1, 0] - p[-1, 1]
    for k, x in ((2, v.double()), (6, (gx * gx + gy * gy).double().sqrt())):
        mean = total(x) / n
        f[:, k], f[:, k + 1] = mean, (total((x - mean[obj]) ** 2) / n).sqrt()
        f[:, k + 2], f[:, k + 3] = extreme(x, "amin"), extreme(x, "amax")
    i, j = [t.double() for t in torch.meshgrid(torch.arange(8, device="cuda"), torch.arange(8, device="cuda"), indexing="ij")]
    i, j, used = i.reshape(-1), j.reshape(-1), torch.zeros(K, dtype=torch.float64, device="cuda")
    for dx, dy in ((1, 0), (0, 1), (1, 1), (1, -1)):
        pair = same(dy, dx)
        key = (obj * 64 + (v >> 5) * 8 + (at(hem, dy, dx) >> 5))[pair]
        c = torch.bincount(key, minlength=K * 64).view(K, 64).double()
        t = c.sum(1)
        some = t > 0
        q = c / t.clamp(min=1)[:, None]
        used += some
        f[:, 10] += ((i - j) ** 2 * q).sum(1)
        f[:, 11] += (q * q).sum(1)
        f[:, 12] += (q / (1 + (i - j) ** 2)).sum(1)
        f[:, 13] += torch.where(q > 0, -q * torch.log(torch.where(q > 0, q, torch.ones_like(q))), torch.zeros_like(q)).sum(1)
        # moments as whole numbers, so that a constant marginal has variance 0
        si, sj = (c * i).sum(1), (c * j).sum(1)
        vi, vj = t * (c * i * i).sum(1) - si * si, t * (c * j * j).sum(1) - sj * sj
        ok = (vi > 0) & (vj > 0)
        f[:, 14] += torch.where(ok, (t * (c * i * j).sum(1) - si * sj) / torch.where(ok, vi * vj, torch.ones_like(vi)).sqrt(), torch.zeros_like(vi))
    f[:, 10:] /= used.clamp(min=1)[:, None]
    return f


def exact(case, seed):
    """The feature rows in 64 bits; the planes are whole numbers, and so is all that the other kinds give."""
    if case["kind"] not in ("plain", "batch", "served"):
        return None
    feats = []
    for rgb in _images(case, seed):
        hem = _exact_hem8(rgb)
        labels, K = _exact_labels(hem)
        feats.append(_exact_features(hem, labels, K))
    if case["kind"] == "served":
        rows = np.zeros((case["n"], _rows(case["W"], case["H"]), P.NFEAT))
        for i, f in enumerate(feats):
            rows[i, :f.shape[0]] = f.cpu().numpy()
        return dict(n_objects=None, status=None, feats=rows)
    rows = []
    for f, (W, H, _, _) in zip(feats, _tiles(case)):
        rows.append(torch.zeros(_rows(W, H), P.NFEAT, dtype=torch.float64, device="cuda"))
        rows[-1][:f.shape[0]] = f
    return dict(hem8=None, labels=None, edt=None, n_objects=None, feats=torch.cat(rows))
