"""What is timed of this package: the calls an EBSD indexing program makes, over the sizes it makes them at.

A case is one kind of call with its sizes:

    index      xcf_index: the library search of one map (or of a few points of it)
    prep       xcf_prep: spectra and filtered images of a batch of patterns
    library    xcf_build_library: the templates of a phase, once per map or pattern centre
    refine     xcf_refine: orientation refinement from seeds near the truth
    precision  xcf_index_precision: tensor-core screen, FP32 rescore, refinement
    maps       xcf_index_maps: several maps of uneven detectors in one captured launch
    learned    xcf_index_learned: network proposals, scored and refined, full search as fallback
    train      xcf_net_loss_grad: one training step's loss and gradient
    ndp        xcf_index_ndp: dictionary indexing by the normalised dot product

Patterns are projections of a band master pattern at known orientations with Poisson counts on a
background, made here with torch (no kernel of the package makes an input).  Orientations that a call
returns in float64 are compared in float32, the precision a map file stores them in.
"""
import functools
import math

import torch

import paper_1807_11313_gb300 as px

PC = (0.5, 0.5, 0.6)
TILT = 70.0
SIDES = (16, 32, 64, 96, 128, 160, 200, 256)
DEV = "cuda"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # 16 points against a small library of 64 px templates: interactive use, one call per few points
        dict(name="index_64_few", kind="index", w=64, h=64, T=300, P=16, native=0, pcs=0),
        # the plain search of a map: 128 px patterns, a 5.35 degree cubic library
        dict(name="index_128_map", kind="index", w=128, h=128, T=4065, P=2000, native=0, pcs=1),
        # the same at 256 px, cropped from an uneven detector, with a coarse library
        dict(name="index_256_map", kind="index", w=275, h=261, T=1018, P=300, native=0, pcs=1),
        # a 160 px detector used whole (mixed-radix sides)
        dict(name="index_160_native", kind="index", w=168, h=160, T=1018, P=301, native=1, pcs=0),
        # pre-processing a map's patterns before anything else is done with them
        dict(name="prep_128_map", kind="prep", w=128, h=128, P=4999, native=0),
        # the template library of a phase
        dict(name="library_128", kind="library", w=128, h=128, T=4065),
        # refinement of a map from its best templates, per-pattern pattern centres
        dict(name="refine_128_map", kind="refine", w=128, h=128, P=1999),
        # 256 px patterns against a 20,000-template library by screen, rescore and refinement
        dict(name="precision_256", kind="precision", w=256, h=256, T=19944, P=1000, k=32),
        # three maps of uneven detectors and libraries, captured once and replayed
        dict(name="maps_96_128_160", kind="maps", w0=96, T0=1018, P0=2000, w1=128, T1=2030, P1=400, w2=160, T2=4065, P2=300),
        # a map by network proposals; one pattern in 50 belongs to a grain the network does not know
        dict(name="learned_128", kind="learned", w=128, h=128, T=4065, P=2000, heads=8),
        # one training batch of the proposal network
        dict(name="train_128", kind="train", B=256, heads=8),
        # dictionary indexing against a fine library
        dict(name="ndp_128", kind="ndp", w=128, h=128, T=39784, P=2000, k=4),
    ]


def _pair_flops(n):
    return 2.5 * n * n * math.log2(n * n) + 6.0 * n * (n // 2 + 1)


def _spread(rng, lo, hi):
    """A whole number of [lo, hi], even over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _detector(rng, n):
    """A detector whose crop has side n, now and then uneven."""
    top = {16: 31, 32: 63, 64: 127, 128: 255}.get(n, n + 40)
    if rng.random() < 0.5:
        return n, n
    return rng.randint(n, min(top, n + 40)), rng.randint(n, min(top, n + 40))


def draw(rng):
    kind = rng.choice(["index", "index", "index", "prep", "library", "refine", "precision", "maps", "learned", "train", "ndp"])
    most = 2000 * 4065 * _pair_flops(128)
    if kind == "index":
        n = rng.choice(SIDES)
        native = 1 if n in (96, 160, 200) else 0
        w, h = (n + rng.randint(0, 15), n + rng.randint(0, 15)) if native else _detector(rng, n)
        T = _spread(rng, 100, 20000)
        # the slower sides take fewer pairs, so that no drawn case is dearer than the largest listed one
        rate = 1.0 if n == 128 else 0.2
        return dict(kind=kind, w=w, h=h, T=T, P=_spread(rng, 1, max(1, min(2500, int(rate * most / _pair_flops(n) / T)))), native=native, pcs=rng.randint(0, 1))
    if kind == "prep":
        n = rng.choice(SIDES)
        native = 1 if n in (96, 160, 200) else 0
        w, h = (n + rng.randint(0, 15), n + rng.randint(0, 15)) if native else _detector(rng, n)
        return dict(kind=kind, w=w, h=h, P=_spread(rng, 1, min(5000, (1 << 27) // (n * n))), native=native)
    if kind == "library":
        n = rng.choice((64, 128, 256))
        w, h = _detector(rng, n)
        return dict(kind=kind, w=w, h=h, T=_spread(rng, 100, {64: 10000, 128: 8000, 256: 2500}[n]))
    if kind == "refine":
        n = rng.choice((64, 128, 128, 256))
        w, h = _detector(rng, n)
        return dict(kind=kind, w=w, h=h, P=_spread(rng, 1, {64: 4000, 128: 3000, 256: 800}[n]))
    if kind == "precision":
        n = rng.choice((128, 256))
        w, h = _detector(rng, n)
        return dict(kind=kind, w=w, h=h, T=_spread(rng, 1000, 20000), P=_spread(rng, 1, 1200), k=rng.randint(4, 32))
    if kind == "maps":
        c = dict(kind=kind)
        for i in range(3):
            w = rng.choice((64, 96, 128, 160, 200))
            c["w%d" % i], c["T%d" % i] = w, _spread(rng, 300, 4000)
            c["P%d" % i] = _spread(rng, 1, max(1, min(2000, int(0.1 * most / _pair_flops(64 if w < 128 else 128) / c["T%d" % i]))))
        return c
    if kind == "learned":
        w, h = _detector(rng, 128)
        return dict(kind=kind, w=w, h=h, T=_spread(rng, 300, 5000), P=_spread(rng, 1, 2500), heads=rng.choice((4, 8, 12)))
    if kind == "train":
        return dict(kind=kind, B=_spread(rng, 16, 512), heads=rng.choice((4, 8, 12)))
    n = rng.choice((64, 128, 256))
    w, h = _detector(rng, n)
    return dict(kind=kind, w=w, h=h, T=_spread(rng, 1000, {64: 40000, 128: 40000, 256: 10000}[n]), P=_spread(rng, 1, {64: 4000, 128: 3000, 256: 600}[n]), k=rng.randint(1, 8))


# ------------------------------------------------------------------ inputs
#: (plane family, weight) of a body-centred cubic crystal; the band half-width grows as 1 / d from 1.5 degrees
BANDS = (((1, 1, 0), 1.0), ((2, 0, 0), 0.9), ((2, 1, 1), 0.8), ((2, 2, 0), 0.7), ((3, 1, 0), 0.6))
MASTER_SIDE = 1024


@functools.lru_cache(maxsize=2)
def _master():
    """[2, M, M] float32: sech^2 bands on the great circles of the plane normals, on the equal-area square grid."""
    M = MASTER_SIDE
    half = math.sqrt(math.pi / 2.0)
    c = half * (2.0 * (torch.arange(M, dtype=torch.float64, device=DEV) + 0.5) / M - 1.0)
    Y, X = torch.meshgrid(c, c, indexing="ij")
    swap = Y.abs() > X.abs()
    a, b = torch.where(swap, Y, X), torch.where(swap, X, Y)
    f = (2.0 * a / math.pi) * torch.sqrt(torch.clamp(math.pi - a * a, min=0.0))
    ang = math.pi * b / (4.0 * torch.where(a == 0, torch.ones_like(a), a))
    u, v = f * torch.cos(ang), f * torch.sin(ang)
    north = torch.stack([torch.where(swap, v, u), torch.where(swap, u, v), 1.0 - 2.0 * a * a / math.pi], dim=-1)
    dirs = torch.stack([north, north * torch.tensor([1.0, 1.0, -1.0], dtype=torch.float64, device=DEV)])
    out = torch.full(dirs.shape[:3], 0.25, dtype=torch.float64, device=DEV)
    for hkl, weight in BANDS:
        seen = set()
        for i in range(6):
            p = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))[i]
            for s in range(8):
                n = tuple(hkl[p[j]] * (1 - 2 * ((s >> j) & 1)) for j in range(3))
                seen.add(max(n, tuple(-x for x in n)))
        length = math.sqrt(sum(x * x for x in hkl))
        sigma = math.radians(1.5) * length / math.sqrt(2.0)
        for n in sorted(seen):
            dot = (dirs @ torch.tensor(n, dtype=torch.float64, device=DEV)) / length
            t = torch.clamp(torch.asin(torch.clamp(dot, -1.0, 1.0)) / sigma, -40.0, 40.0)
            out += weight / torch.cosh(t) ** 2
    return out.float().contiguous()


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(shape, g, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(shape, generator=g, dtype=torch.float64, device=DEV)


def _canon(q):
    q = q / q.norm(dim=-1, keepdim=True)
    return torch.where(q[..., :1] < 0, -q, q).contiguous()


def _quats(n, g):
    """n uniformly random orientations."""
    u = _rand((3, n), g)
    r1, r2, t1, t2 = torch.sqrt(1 - u[0]), torch.sqrt(u[0]), 2 * math.pi * u[1], 2 * math.pi * u[2]
    return _canon(torch.stack([r2 * torch.cos(t2), r1 * torch.sin(t1), r1 * torch.cos(t1), r2 * torch.sin(t2)], dim=-1))


def _qmul(a, b):
    aw, ax, ay, az = a.unbind(-1)
    bw, bx, by, bz = b.unbind(-1)
    return torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                        aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], dim=-1)


def _near(q, deg, g):
    """q turned by up to `deg` degrees about each axis."""
    v = _rand((q.shape[0], 3), g, -math.radians(deg), math.radians(deg))
    t = v.norm(dim=-1, keepdim=True)
    return _canon(_qmul(q, torch.cat([torch.cos(t / 2), torch.sin(t / 2) * v / t.clamp(min=1e-30)], dim=-1)))


def _pcs(n, g):
    return (torch.tensor(PC, dtype=torch.float64, device=DEV) + _rand((n, 3), g, -0.005, 0.005)).contiguous()


def _matrix(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], dim=-1).reshape(-1, 3, 3)


def _project(q, pcs, w, h, dtype=torch.float32, most=1 << 25):
    """Gnomonic projections [P, h, w] of the master at orientations q and pattern centres pcs (None: PC)."""
    M, m = MASTER_SIDE, _master().to(dtype).reshape(-1)
    P, out = q.shape[0], torch.empty((q.shape[0], h, w), dtype=dtype, device=DEV)
    a = math.radians(90.0 - TILT)
    tilt = torch.tensor([[1, 0, 0], [0, math.cos(a), -math.sin(a)], [0, math.sin(a), math.cos(a)]], dtype=torch.float64, device=DEV)
    x = torch.arange(w, dtype=dtype, device=DEV) + 0.5
    y = torch.arange(h, dtype=dtype, device=DEV) + 0.5
    step = max(1, most // (w * h))
    for p in range(0, P, step):
        G = (_matrix(q[p:p + step].double()) @ tilt).to(dtype)
        pc = (torch.tensor(PC, dtype=torch.float64, device=DEV).expand(G.shape[0], 3) if pcs is None else pcs[p:p + step]).to(dtype)
        dx = (x - pc[:, :1] * w)[:, None, :]
        dy = (pc[:, 1:2] * h - y)[:, :, None]
        dz = (pc[:, 2] * w)[:, None, None]
        r = torch.rsqrt(dx * dx + dy * dy + dz * dz) if dtype == torch.float32 else 1.0 / torch.sqrt(dx * dx + dy * dy + dz * dz)
        d = [(G[:, i, 0, None, None] * dx + G[:, i, 1, None, None] * dy + G[:, i, 2, None, None] * dz) * r for i in range(3)]
        s2 = d[0] * d[0] + d[1] * d[1]
        qv = torch.sqrt(2.0 * s2 / (1.0 + d[2].abs()))
        big = d[1].abs() <= d[0].abs()
        num, den = torch.where(big, d[1], d[0]), torch.where(big, d[0], d[1])
        den = torch.where(den == 0, torch.full_like(den, 1e-30), den)
        sg = torch.where(den >= 0, 1.0, -1.0).to(dtype)
        u, t = sg * qv * (math.sqrt(math.pi) / 2), sg * qv * (2 / math.sqrt(math.pi)) * torch.atan(num / den)
        X, Y = torch.where(big, u, t), torch.where(big, t, u)
        inv = 1.0 / math.sqrt(math.pi / 2)
        fx = ((X * inv + 1) * (0.5 * M) - 0.5).clamp(0, M - 1)
        fy = ((Y * inv + 1) * (0.5 * M) - 0.5).clamp(0, M - 1)
        i0, j0 = fx.floor().long().clamp(max=M - 2), fy.floor().long().clamp(max=M - 2)
        tx, ty = fx - i0, fy - j0
        o = torch.where(d[2] >= 0, 0, M * M) + j0 * M + i0
        out[p:p + step] = (1 - ty) * ((1 - tx) * m[o] + tx * m[o + 1]) + ty * ((1 - tx) * m[o + M] + tx * m[o + M + 1])
    return out


def _patterns(q, pcs, w, h, g, lo=100.0, hi=100.0):
    """Poisson counts of the projections on a Gaussian background, peak counts in [lo, hi]."""
    clean = _project(q, pcs, w, h)
    P = q.shape[0]
    pc = (torch.tensor(PC, dtype=torch.float64, device=DEV).expand(P, 3) if pcs is None else pcs).float()
    peak = _rand((P, 1, 1), g, lo, hi).float()
    x, y = torch.arange(w, device=DEV) + 0.5, torch.arange(h, device=DEV) + 0.5
    s2 = 2 * (0.35 * w) ** 2
    for p in range(0, P, 2048):
        c = clean[p:p + 2048]
        c = (c - c.amin((1, 2), keepdim=True)) / (c.amax((1, 2), keepdim=True) - c.amin((1, 2), keepdim=True))
        b = torch.exp(-((y[:, None] - pc[p:p + 2048, 1, None, None] * h) ** 2 + (x - pc[p:p + 2048, 0, None, None] * w) ** 2) / s2)
        clean[p:p + 2048] = torch.poisson(peak[p:p + 2048] * (0.6 * b + 0.4 * c), generator=g)
    return clean


#: widths of the proposal network's five convolutions and of its hidden layer
CHANNELS, HIDDEN = (1, 32, 64, 64, 128, 128), 256


def _net_blocks(heads, g):
    """Parameter blocks in the network's order, as a new network starts."""
    blocks = []
    for i in range(5):
        fan = CHANNELS[i] * 9
        blocks.append(_rand((CHANNELS[i + 1], CHANNELS[i], 3, 3), g, -1, 1) * math.sqrt(6 / fan))
        blocks.append(torch.full((CHANNELS[i + 1],), 0.01, dtype=torch.float64, device=DEV))
    for rows, cols in ((HIDDEN, CHANNELS[5]), (6 * heads, HIDDEN)):
        blocks.append(_rand((rows, cols), g, -1, 1) * math.sqrt(6 / cols))
        blocks.append(torch.full((rows,), 0.01 if rows == HIDDEN else 0.0, dtype=torch.float64, device=DEV))
    return blocks


def _knowing_net(heads, grains, g):
    """A network whose heads propose the orientations of `grains` (as one trained on those would)."""
    blocks = _net_blocks(heads, g)
    R = _matrix(grains)
    blocks[-2] = torch.zeros_like(blocks[-2])
    blocks[-1] = torch.cat([R[:, :, 0], R[:, :, 1]], dim=1).reshape(-1)
    return torch.cat([b.reshape(-1) for b in blocks]).float().contiguous()


def _inputs(c, seed):
    """The plain tensors of a case: no handle of the package among them."""
    g, k = _gen(seed), c["kind"]
    if k == "maps":
        s = dict(maps=[])
        for i in range(3):
            lib_q = _quats(c["T%d" % i], g)
            w = c["w%d" % i]
            s["maps"].append(dict(lib_q=lib_q, templates=_project(lib_q, None, w, w), pats=_patterns(_quats(c["P%d" % i], g), None, w, w, g, 50, 500)))
        return s
    if k == "train":
        q = _quats(c["B"], g)
        pats = _patterns(q, _pcs(c["B"], g), 128, 128, g, 50, 500)
        return dict(q=q, pats=pats, blocks=[b.float() for b in _net_blocks(c["heads"], g)])
    w, h = c["w"], c["h"]
    if k == "library":
        return dict(lib_q=_quats(c["T"], g))
    if k == "prep":
        return dict(pats=_patterns(_quats(c["P"], g), _pcs(c["P"], g), w, h, g, 50, 500))
    if k == "index":
        lib_q = _quats(c["T"], g)
        pcs = _pcs(c["P"], g) if c["pcs"] else None
        return dict(lib_q=lib_q, templates=_project(lib_q, None, w, h), pcs=pcs, pats=_patterns(_quats(c["P"], g), pcs, w, h, g))
    pcs = _pcs(c["P"], g)
    if k == "learned":
        grains = _quats(c["heads"], g)
        truth = _near(grains[torch.arange(c["P"], device=DEV) % c["heads"]], 2.0, g)
        stray = torch.arange(c["P"], device=DEV) % 50 == 17
        truth[stray] = _quats(c["P"], g)[stray]
        return dict(lib_q=_quats(c["T"], g), grains=grains, params=_knowing_net(c["heads"], grains, g), pcs=pcs, pats=_patterns(truth, pcs, w, h, g, 100, 500))
    truth = _quats(c["P"], g)
    s = dict(pcs=pcs, pats=_patterns(truth, pcs, w, h, g, 100, 500))
    if k == "refine":
        s["seeds"] = _near(truth, 2.0, g)
    else:
        s["lib_q"] = _quats(c["T"], g)
    return s


#: refined peak below which the learned form falls back to the full search
TAU = 0.15


def prepare(case, seed):
    c = dict(case)
    s = dict(c=c, **_inputs(c, seed))
    k, m = c["kind"], _master()
    s["ctx"] = px.Context(native_sizes=c.get("native", 0))
    if k == "maps":
        s["ctx"].close()
        s["ctx"] = px.Context()
        for d in s["maps"]:
            w = d["pats"].shape[-1]
            d["lib"] = px.xcf_build_library_images(s["ctx"], d.pop("templates"), d["lib_q"], px.geometry(w, w, PC))
        s["outs"] = [(torch.empty(d["pats"].shape[0], dtype=torch.int32, device=DEV), torch.empty(d["pats"].shape[0], device=DEV),
                      torch.empty((d["pats"].shape[0], 2), device=DEV)) for d in s["maps"]]
        return s
    if k == "train":
        s["net"] = px.xcf_net_create(s["ctx"], c["heads"], torch.cat([b.reshape(-1) for b in s.pop("blocks")]).contiguous())
        return s
    s["geom"] = px.geometry(c["w"], c["h"], PC)
    if k == "index":
        s["lib"] = px.xcf_build_library_images(s["ctx"], s.pop("templates"), s["lib_q"], s["geom"])
    elif k == "refine":
        s["lib"] = px.xcf_build_library(s["ctx"], m, s["seeds"][:1].contiguous(), s["geom"])
    elif k == "precision":
        s["lib"] = px.xcf_build_library_ex(s["ctx"], s["lib_q"], s["geom"], master=m, flags=px.XCF_LIB_SCREEN)
    elif k == "learned":
        s["lib"] = px.xcf_build_library(s["ctx"], m, s["lib_q"], s["geom"])
        s["net"] = px.xcf_net_create(s["ctx"], c["heads"], s["params"])
        s["net"].set_bf16(True)
    elif k == "ndp":
        s["lib"] = px.xcf_build_library_ex(s["ctx"], s["lib_q"], s["geom"], master=m, flags=px.XCF_LIB_NDP | px.XCF_LIB_NO_SPECTRA)
    return s


# ------------------------------------------------------------------ the calls
def run(s):
    c, ctx = s["c"], s["ctx"]
    k = c["kind"]
    if k == "index":
        best, peak, shift = px.xcf_index(ctx, s["lib"], s["pats"], pcs=s["pcs"])
        return dict(best=best, peak=peak, shift=shift)
    if k == "prep":
        spectra, spatial, degenerate = px.xcf_prep(ctx, s["pats"], s["geom"], want_spatial=True)
        return dict(spectra=spectra, spatial=spatial, degenerate=degenerate)
    if k == "library":
        return dict(spectra=px.xcf_build_library(ctx, _master(), s["lib_q"], s["geom"]).spectra())
    if k == "refine":
        q, peak, iters = px.xcf_refine(ctx, s["lib"], s["pats"], s["seeds"], pcs=s["pcs"])
        return dict(quats=q.float(), peak=peak, iters=iters)
    if k == "precision":
        best, q, peak, iters = px.xcf_index_precision(ctx, s["lib"], s["pats"], pcs=s["pcs"], k=c["k"])
        return dict(best=best, quats=q.float(), peak=peak, iters=iters)
    if k == "maps":
        px.xcf_index_maps(ctx, [(d["lib"], d["pats"]) for d in s["maps"]], outs=s["outs"], graph=True)
        return [dict(best=b, peak=p, shift=t) for b, p, t in s["outs"]]
    if k == "learned":
        q, peak, iters, fallback = px.xcf_index_learned(ctx, s["net"], s["lib"], s["pats"], pcs=s["pcs"], tau=TAU)
        return dict(quats=q.float(), peak=peak, iters=iters, fallback=fallback)
    if k == "train":
        loss, grad, winners = px.xcf_net_loss_grad(ctx, s["net"], s["pats"], s["q"], want_grad=True, want_winners=True)
        return dict(loss=loss.float(), grad=grad, winners=winners)
    best, ndp = px.xcf_index_ndp(ctx, s["lib"], s["pats"], k=c["k"])
    return dict(best=best, ndp=ndp)


def _side(c):
    m = min(c["w"], c["h"])
    return max(n for n in (SIDES if c.get("native") else (16, 32, 64, 128, 256)) if n <= m)


def work(case):
    c = case
    k = c["kind"]
    if k == "train":
        macs, S = 0, 128
        for i in range(5):
            S //= 2
            macs += S * S * CHANNELS[i + 1] * CHANNELS[i] * 9
        macs += CHANNELS[5] * HIDDEN + HIDDEN * 6 * c["heads"]
        n = sum(CHANNELS[i + 1] * (CHANNELS[i] * 9 + 1) for i in range(5)) + HIDDEN * (CHANNELS[5] + 1) + 6 * c["heads"] * (HIDDEN + 1)
        # forward, and backward to the weights and to every layer's input but the first
        return dict(bytes=4 * c["B"] * 128 * 128 + 8 * n, flops=2.0 * c["B"] * (3 * macs - 64 * 64 * 32 * 9))
    if k == "maps":
        b = f = 0.0
        for i in range(3):
            w = c["w%d" % i]
            n = _side(dict(w=w, h=w))
            T, P = c["T%d" % i], c["P%d" % i]
            b += 4.0 * P * w * w + 8.0 * T * n * (n // 2 + 1) + 16 * P
            f += P * T * _pair_flops(n)
        return dict(bytes=b, flops=f)
    n = _side(c)
    half, image, fft = 8.0 * n * (n // 2 + 1), 4.0 * c["w"] * c["h"], 2.5 * n * n * math.log2(n * n)
    P, T = c.get("P", 0), c.get("T", 0)
    if k == "index":
        return dict(bytes=P * image + T * half + 16 * P, flops=P * (T * _pair_flops(n) + fft))
    if k == "prep":
        return dict(bytes=P * (image + half + 4.0 * n * n), flops=2.0 * P * fft)
    if k == "library":
        # each spectrum written once and copied out once
        return dict(bytes=8.0 * MASTER_SIDE ** 2 + 32 * T + 3 * T * half, flops=T * (fft + 60.0 * n * n))
    # one refinement iteration: two projected templates transformed, one correlation, one template transformed back
    it = 2 * (60.0 * n * n + fft) + _pair_flops(n) + fft
    if k == "refine":
        return dict(bytes=P * (image + 100) + 8.0 * MASTER_SIDE ** 2, flops=P * (2 * it + 2 * fft))
    if k == "precision":
        return dict(bytes=P * image + 2.0 * T * n * n + P * c["k"] * half, flops=P * (2.0 * T * n * n + c["k"] * _pair_flops(n) + 2 * it + 2 * fft))
    if k == "learned":
        return dict(bytes=P * image + 8.0 * MASTER_SIDE ** 2, flops=P * (73.2e6 + c["heads"] * (60.0 * n * n + fft + _pair_flops(n)) + 2 * it + 2 * fft + T * _pair_flops(n) / 50))
    return dict(bytes=P * image + 2.0 * T * n * n, flops=2.0 * P * T * n * n)


# ------------------------------------------------------------------ the same in 64 bits
def _crop(c):
    n = _side(c)
    ox, oy = (c["w"] - n) // 2, (c["h"] - n) // 2
    return n, ox, oy


def _band(n):
    f = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=DEV)
    r2 = f[:, None] ** 2 + torch.arange(n // 2 + 1, dtype=torch.float64, device=DEV) ** 2
    return -torch.expm1(-r2 / 8.0) * torch.exp(-r2 / (2.0 * (n / 4.0) ** 2))


def _spectra64(img):
    """Unit-norm filtered half spectra of square images [P, n, n]."""
    n = img.shape[-1]
    out = torch.empty((img.shape[0], n, n // 2 + 1), dtype=torch.complex128, device=DEV)
    win = 0.5 - 0.5 * torch.cos(2 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n)
    weight = torch.full((n // 2 + 1,), 2.0, dtype=torch.float64, device=DEV)
    weight[0] = weight[-1] = 1.0
    for p in range(0, img.shape[0], 1024):
        x = img[p:p + 1024].double()
        x = (x - x.mean((1, 2), keepdim=True)) / x.std((1, 2), keepdim=True, unbiased=False)
        S = torch.fft.rfft2(x * win * win[:, None]) * _band(n)
        out[p:p + 1024] = S / torch.sqrt((S.abs() ** 2 * weight).sum((1, 2), keepdim=True))
    return out


def _spatial64(S):
    n = S.shape[1]
    return torch.cat([torch.fft.irfft2(S[p:p + 1024], s=(n, n), norm="ortho") for p in range(0, S.shape[0], 1024)])


def _fit(m, z, p):
    den = m - 2 * z + p
    return torch.where(den < 0, ((m - p) / (2 * torch.where(den < 0, den, torch.ones_like(den)))).clamp(-0.5, 0.5), torch.zeros_like(den))


def _peak64(St, Sp):
    """Integer peak and parabolic shift of each pair's surface."""
    n, peaks, shifts = Sp.shape[1], [], []
    for p in range(0, Sp.shape[0], 512):
        r = torch.fft.irfft2(St[p:p + 512].conj() * Sp[p:p + 512], s=(n, n), norm="forward")
        top, i = r.flatten(1).max(1)
        y, x, b = i // n, i % n, torch.arange(r.shape[0], device=DEV)
        at = lambda dy, dx: r[b, (y + dy) % n, (x + dx) % n]  # noqa: E731
        dx = torch.where(x < n // 2, x, x - n) + _fit(at(0, -1), top, at(0, 1))
        dy = torch.where(y < n // 2, y, y - n) + _fit(at(-1, 0), top, at(1, 0))
        peaks.append(top)
        shifts.append(torch.stack([dx, dy], dim=1))
    return torch.cat(peaks), torch.cat(shifts)


def _search64(St, Sp, cand=None):
    """Best template of each pattern: a first look in 32 bits, then every template within 1e-4 of it in 64."""
    n, best = Sp.shape[1], []
    t32, step = (St.to(torch.complex64) if cand is None else None), max(1, (1 << 28) // (n * n))
    for p in range(Sp.shape[0]):
        T = St if cand is None else St[cand[p]]
        low = t32 if cand is None else T.to(torch.complex64)
        s = Sp[p].to(torch.complex64)
        top = torch.cat([torch.fft.irfft2(low[t:t + step].conj() * s, s=(n, n), norm="forward").flatten(1).amax(1) for t in range(0, T.shape[0], step)])
        near = torch.nonzero(top >= top.max() * (1 - 1e-4)).flatten()
        high = torch.fft.irfft2(T[near].conj() * Sp[p], s=(n, n), norm="forward").flatten(1).amax(1)
        t = near[high.argmax()]
        best.append(t if cand is None else cand[p][t])
    return torch.stack(best)


def _turn(q, R):
    a = math.radians(90.0 - TILT) / 2
    qs = torch.tensor([math.cos(a), math.sin(a), 0.0, 0.0], dtype=torch.float64, device=DEV).expand_as(q)
    inv = torch.tensor([1.0, -1.0, -1.0, -1.0], dtype=torch.float64, device=DEV)
    return _canon(_qmul(_qmul(_qmul(q, qs), R * inv), qs * inv))


def _templates64(c, q, pcs):
    n, ox, oy = _crop(c)
    return _spectra64(_project(q, pcs, c["w"], c["h"], torch.float64, 1 << 24)[:, oy:oy + n, ox:ox + n])


def _polar(y):
    """Log-polar images [P, n / 4, 2 n] about the centre."""
    n = y.shape[-1]
    nr, na = n // 4, 2 * n
    lo, hi = n / 4.0, n / 2.0 - 1.0
    r = lo * (hi / lo) ** (torch.arange(nr, dtype=torch.float64, device=DEV) / (nr - 1))
    t = 2 * math.pi * torch.arange(na, dtype=torch.float64, device=DEV) / na
    fx, fy = 0.5 * n - 0.5 + r[:, None] * torch.cos(t), 0.5 * n - 0.5 - r[:, None] * torch.sin(t)
    x0, y0 = fx.floor().long().clamp(0, n - 2), fy.floor().long().clamp(0, n - 2)
    tx, ty = fx - x0, fy - y0
    return (1 - ty) * ((1 - tx) * y[:, y0, x0] + tx * y[:, y0, x0 + 1]) + ty * ((1 - tx) * y[:, y0 + 1, x0] + tx * y[:, y0 + 1, x0 + 1])


def _refine64(c, Sp, seeds, pcs):
    """Two iterations of the refinement, 512 patterns at a time."""
    n = _side(c)
    windows, nr, na = 4, n // 4, 2 * n
    quats, peaks = [], []
    for p in range(0, Sp.shape[0], 512):
        S, q, pc = Sp[p:p + 512], seeds[p:p + 512].double(), pcs[p:p + 512]
        lp = _polar(_spatial64(S))
        for _ in range(2):
            peak, shift = _peak64(_templates64(c, q, pc), S)
            L = pc[:, 2] * c["w"]
            tx, ty = torch.atan(shift[:, 1] / L) / 2, torch.atan(shift[:, 0] / L) / 2
            z = torch.zeros_like(tx)
            q = _turn(q, _qmul(torch.stack([torch.cos(tx), torch.sin(tx), z, z], -1), torch.stack([torch.cos(ty), z, torch.sin(ty), z], -1)))
            lt, found = _polar(_spatial64(_templates64(c, q, pc))), []
            for b in range(windows):
                a0, a1 = b * nr // windows, (b + 1) * nr // windows
                A, B = (torch.fft.rfft(x[:, a0:a1] - x[:, a0:a1].mean((1, 2), keepdim=True)) for x in (lt, lp))
                r = torch.fft.irfft((A.conj() * B).sum(1), n=na)
                top, i = r.max(1)
                rows = torch.arange(r.shape[0], device=DEV)
                found.append(torch.where(i < na // 2, i, i - na) + _fit(r[rows, (i - 1) % na], top, r[rows, (i + 1) % na]))
            mid = torch.stack(found).sort(0).values
            tz = 0.5 * (mid[1] + mid[2]) * math.pi / na
            q = _turn(q, torch.stack([torch.cos(tz), z, z, torch.sin(tz)], -1))
        quats.append(q)
        peaks.append(peak)
    return torch.cat(quats), torch.cat(peaks)


def _loss64(s, heads):
    """Loss and gradient of the proposal network by torch's autograd in float64."""
    blocks = [b.double().requires_grad_() for b in s["blocks"]]
    x = s["pats"].double()
    x = ((x - x.mean((1, 2), keepdim=True)) / x.std((1, 2), keepdim=True, unbiased=False))[:, None]
    for i in range(5):
        x = torch.relu(torch.nn.functional.conv2d(x, blocks[2 * i], blocks[2 * i + 1], stride=2, padding=1))
    x = torch.relu(x.mean((2, 3)) @ blocks[10].T + blocks[11])
    o = (x @ blocks[12].T + blocks[13]).reshape(-1, heads, 2, 3)
    b1 = o[:, :, 0] / o[:, :, 0].norm(dim=-1, keepdim=True)
    b2 = o[:, :, 1] - (b1 * o[:, :, 1]).sum(-1, keepdim=True) * b1
    b2 = b2 / b2.norm(dim=-1, keepdim=True)
    R = torch.stack([b1, b2, torch.cross(b1, b2, dim=-1)], dim=-1)
    ops = []
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        for sg in range(8):
            m = torch.zeros(3, 3, dtype=torch.float64)
            for j in range(3):
                m[j, p[j]] = 1 - 2 * ((sg >> j) & 1)
            if torch.det(m) > 0:
                ops.append(m.to(DEV))
    target = torch.stack(ops)[None] @ _matrix(s["q"])[:, None]
    d = ((R[:, :, None] - target[:, None]) ** 2).sum((3, 4)).flatten(1).amin(1)
    loss = d.mean()
    loss.backward()
    return loss.detach().reshape(1), torch.cat([b.grad.reshape(-1) for b in blocks])


def _blur_norm(x):
    """Background-corrected, standardised images: minus a Gaussian blur of n / 8 px with repeated edges."""
    n = x.shape[-1]
    sigma = n / 8.0
    r = int(round(3 * sigma))
    k = torch.exp(-torch.arange(-r, r + 1, dtype=torch.float64, device=DEV) ** 2 / (2 * sigma * sigma))
    k = k / k.sum()
    at = torch.arange(n, device=DEV)[:, None] + torch.arange(-r, r + 1, device=DEV)
    B = torch.zeros((n, n), dtype=torch.float64, device=DEV).scatter_add_(1, at.clamp(0, n - 1), k.expand(n, -1).contiguous())
    x = x.double()
    x = x - B @ x @ B.T
    return (x - x.mean((1, 2), keepdim=True)) / x.std((1, 2), keepdim=True, unbiased=False)


def exact(case, seed):
    c = dict(case)
    s, k = _inputs(c, seed), c["kind"]
    if k == "train":
        loss, grad = _loss64(s, c["heads"])
        return dict(loss=loss, grad=grad, winners=None)
    if k == "maps":
        out = []
        for d in s["maps"]:
            w = d["pats"].shape[-1]
            n, ox, oy = _crop(dict(w=w, h=w))
            St, Sp = (_spectra64(x[:, oy:oy + n, ox:ox + n]) for x in (d["templates"], d["pats"]))
            peak, shift = _peak64(St[_search64(St, Sp)], Sp)
            out.append(dict(best=None, peak=peak, shift=shift))
        return out
    if k == "library":
        return dict(spectra=_templates64(c, s["lib_q"], None))
    n, ox, oy = _crop(c)
    crops = s["pats"][:, oy:oy + n, ox:ox + n]
    if k == "ndp":
        X = _blur_norm(crops).flatten(1) / n
        top = torch.full((X.shape[0],), -2.0, dtype=torch.float64, device=DEV)
        for t in range(0, c["T"], 2048):
            Y = _blur_norm(_project(s["lib_q"][t:t + 2048], None, c["w"], c["h"], torch.float64, 1 << 24)[:, oy:oy + n, ox:ox + n]).flatten(1) / n
            top = torch.maximum(top, (X @ Y.T).amax(1))
        return dict(best=None, ndp=top)
    Sp = _spectra64(crops)
    if k == "prep":
        return dict(spectra=Sp, spatial=_spatial64(Sp), degenerate=None)
    if k == "index":
        St = _spectra64(s["templates"][:, oy:oy + n, ox:ox + n])
        peak, shift = _peak64(St[_search64(St, Sp)], Sp)
        if s["pcs"] is not None:
            shift = shift - (s["pcs"][:, :2] - torch.tensor(PC[:2], dtype=torch.float64, device=DEV)) * torch.tensor([c["w"], c["h"]], dtype=torch.float64, device=DEV)
        return dict(best=None, peak=peak, shift=shift)
    if k == "refine":
        q, peak = _refine64(c, Sp, s["seeds"], s["pcs"])
        return dict(quats=q, peak=peak, iters=None)
    if k == "precision":
        # the screen only proposes: the best of the k templates nearest at zero shift
        y, score = _spatial64(Sp).flatten(1).float(), []
        for t in range(0, c["T"], 1024):
            score.append(y @ _spatial64(_templates64(c, s["lib_q"][t:t + 1024], None)).flatten(1).float().T)
        cand = torch.cat(score, 1).topk(c["k"], 1).indices
        best = []
        for p in range(c["P"]):
            best.append(_search64(_templates64(c, s["lib_q"][cand[p]], None), Sp[p:p + 1]))
            best[-1] = cand[p][best[-1]]
        q, peak = _refine64(c, Sp, s["lib_q"][torch.cat(best)], s["pcs"])
        return dict(best=None, quats=q, peak=peak, iters=None)
    # learned: the best of the network's proposals, refined; the full search where that stays below TAU
    tops = torch.stack([_peak64(_templates64(c, g[None].expand(c["P"], 4).contiguous(), s["pcs"]), Sp)[0] for g in s["grains"]])
    q, peak = _refine64(c, Sp, s["grains"][tops.argmax(0)], s["pcs"])
    low = torch.nonzero(peak < TAU).flatten()
    if low.numel():
        best = _search64(_templates64(c, s["lib_q"], None), Sp[low])
        q[low], peak[low] = _refine64(c, Sp[low], s["lib_q"][best], s["pcs"][low])
    return dict(quats=q, peak=peak, iters=None, fallback=None)
