"""The work a program gives this library, case by case, through its public
entry points: one formula on one image, big formulas replayed as a batch,
batches of slices, query batches, labelling, volumes.

A case is a dict of plain values.  `prepare` makes its inputs on the GPU from
a seed and keeps what a program keeps between calls (context, compiled
formulas, prepared batch, output buffers); `run` is one pass.  Every output
is a packed mask or a label array: whole numbers.
"""
import math
import random

import numpy as np
import torch

import paper_2010_07284_gb300 as vg

# ------------------------------------------------------------------ specs --
# Specification texts in the command language of the library.

# Reachability past a barrier and a surround test on one smooth image.
BARRIER = """
load x = "x"
let a = intensity(x) >. 0.6
let b = intensity(x) <. 0.3
save "past" rho(N(a), !b) & !a
save "held" surrounded(a, !b)
"""

# The case-study segmentation: very bright seeds grown through bright pixels.
GROW = """
load flair = "flair"
let hi = intensity(flair) >. {hi}
let vi = intensity(flair) >. {vi}
save "gtv" grow(hi, vi)
"""

# A segmentation of 4-channel scans: percentile thresholds, closing, region
# contact, edges (about forty primitive operators).
SEGMENT = """
load s = "scan"
let hi = channel(s, 0) >. percentile(channel(s, 0), 0.95)
let vi = channel(s, 0) >. percentile(channel(s, 0), 0.86)
let gtv = grow(hi, vi)
let rim = channel(s, 1) >. percentile(channel(s, 1), 0.97)
let core = channel(s, 2) >. percentile(channel(s, 2), 0.98)
let brain = channel(s, 3) >. percentile(channel(s, 3), 0.30)
let dark = channel(s, 3) <. 0.08
save "seg" interior(N(N(N(gtv)))) & brain & !dark
save "act" surrounded(core, rim) | touch(rim, core)
save "gtv" gtv
save "edge" gtv & !interior(gtv)
"""

# Channel arithmetic: a normalised difference and a product, cut at
# percentiles, cleaned by contact.
TERMS = """
load s = "pair"
let d = (channel(s, 0) - channel(s, 1)) / (channel(s, 0) + channel(s, 1) + 1)
let m = channel(s, 0) * channel(s, 1)
let up = d >. percentile(d, 0.9)
let big = m >. percentile(m, 0.75)
let low = d <. percentile(d, 0.25)
save "lesion" grow(up & big, big)
save "shell" N(low) & !touch(low, up)
"""


def _random_dag(nodes, seed):
    """A random formula: 35 % thresholds on a U[0, 1) image, 35 % not/and, 20 %
    N, 10 % rho; an operand is mostly one of the last four nodes; depth at most
    min(500, nodes).  Its outputs are the nodes nobody consumes."""
    rng = random.Random(1_000_003 * seed + nodes)
    cap = min(500, nodes)
    out, depth, used = [], [], [False] * nodes
    for i in range(nodes):
        kind = "THR" if i == 0 else rng.choices(("THR", "NOT", "AND", "NEAR", "REACH"),
                                                (35, 17.5, 17.5, 20, 10))[0]
        if kind == "THR":
            out.append((rng.choice(("THR_GT", "THR_LT")), -1, -1, 0, 0, rng.random(), 0.0))
            depth.append(1)
            continue
        arity = 1 if kind in ("NOT", "NEAR") else 2
        while True:
            ops = [rng.randrange(max(0, i - 4), i) if rng.random() < 0.7 else rng.randrange(i)
                   for _ in range(arity)]
            d = 1 + max(depth[k] for k in ops)
            if d <= cap:
                break
        for k in ops:
            used[k] = True
        out.append((kind, ops[0], ops[1] if arity == 2 else -1, 0, 0, 0.0, 0.0))
        depth.append(d)
    return out, [i for i in range(nodes) if not used[i]]


CHAIN_MIXES = {"mixed": (30, 30, 25, 15), "near": (30, 65, 5, 0), "reach": (30, 10, 20, 40)}


def _chain(nodes, seed, mix):
    """A sequential formula f(g(...(x))): every operator takes the previous
    node, binary ones a fresh threshold beside it.  Sixteen states on the way
    are outputs too (the last one alone is often empty or full)."""
    rng = random.Random(7_000_003 * seed + nodes)
    out = [("THR_GT", -1, -1, 0, 0, rng.random(), 0.0)]
    while len(out) < nodes:
        kind = rng.choices(("NOT", "NEAR", "AND", "REACH"), CHAIN_MIXES[mix])[0]
        prev = len(out) - 1
        if kind in ("NOT", "NEAR"):
            out.append((kind, prev, -1, 0, 0, 0.0, 0.0))
        else:
            out.append((rng.choice(("THR_GT", "THR_LT")), -1, -1, 0, 0, rng.random(), 0.0))
            out.append((kind, prev, len(out) - 1, 0, 0, 0.0, 0.0))
    last = len(out) - 1
    return out, sorted({last} | set(range(0, last, max(1, last // 15))))


# ----------------------------------------------------------------- images --

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(c, h, w, g):
    return torch.rand((c, h, w), generator=g, device="cuda", dtype=torch.float32)


def _blur(x, sigma):
    """Separable Gaussian blur, truncated at 3 sigma, reflected border."""
    r = int(3 * sigma + 0.5)
    k = np.exp(-0.5 * (np.arange(-r, r + 1) / sigma) ** 2)
    k = (k / k.sum()).tolist()
    for dim in (-2, -1):
        n = x.shape[dim]
        at = torch.arange(-r, n + r, device=x.device)
        at = torch.where(at < 0, -1 - at, at) % (2 * n)
        at = torch.where(at >= n, 2 * n - 1 - at, at)
        p = x.index_select(dim, at)
        y = torch.zeros_like(x)
        for i, wt in enumerate(k):
            y += wt * p.narrow(dim, i, n)
        x = y
    return x


def _smooth(h, w, g, sigma=4.0):
    """A smooth random field rescaled to [0, 1]."""
    x = _blur(torch.randn((1, h, w), generator=g, device="cuda"), sigma)
    lo, hi = x.min(), x.max()
    return (x - lo) / (hi - lo)


def _phantom(shape, rng, g):
    """A 4-channel scan of `shape` (h, w) or (d, h, w): a brain ellipsoid with
    a bright core, a rim and a halo, and N(0, 0.05) noise on every channel."""
    axes = [torch.arange(n, device="cuda", dtype=torch.float32).reshape(
        [-1 if k == i else 1 for k in range(len(shape))]) for i, n in enumerate(shape)]

    def blob(centre, radii, soft):
        d = sum(((x - c) / r) ** 2 for x, c, r in zip(axes, centre, radii)).sqrt()
        return torch.sigmoid((1.0 - d) / soft)

    mid = [n / 2 + rng.gauss(0, 0.02) * n for n in shape]
    brain = blob(mid, [n * rng.uniform(0.36, 0.44) for n in shape], 0.03)
    at = [n / 2 + rng.uniform(-0.18, 0.18) * n for n in shape]
    rc = min(shape) * rng.uniform(0.05, 0.10)
    ell = [1.0] * (len(shape) - 1) + [rng.uniform(0.7, 1.0)]
    core = blob(at, [rc * e for e in ell], 0.08)
    outer = blob(at, [1.45 * rc * e for e in ell], 0.06)
    rim = (outer - core).clamp(0, 1)
    halo = (blob(at, [2.6 * rc * e for e in ell], 0.15) - outer).clamp(0, 1)
    base = 0.35 * brain
    ch = torch.stack([base + 0.45 * halo + 0.55 * core + 0.30 * rim, base + 0.60 * rim,
                      base + 0.60 * core, 0.30 + 0.40 * brain - 0.20 * (core + rim)])
    return ch + 0.05 * torch.randn(ch.shape, generator=g, device="cuda")


def _upscaled_slice(h, w, rng, g):
    """Channel 0 of a 240 x 240 scan, upscaled bilinearly and clipped to [0, 1]."""
    x = _phantom((240, 240), rng, g)[:1]
    for dim, n in ((1, h), (2, w)):
        at = torch.linspace(0, 239, n, device="cuda")
        lo = at.floor().clamp(max=238).long()
        f = (at - lo).reshape([-1, 1] if dim == 1 else [1, -1])
        x = x.index_select(dim, lo) * (1 - f) + x.index_select(dim, lo + 1) * f
    return x.clamp(0, 1)


def _to_u16(x):
    return (x.clamp(0, 1) * 65535.0).round().to(torch.int32).to(torch.int16).view(torch.uint16)


def _pattern(kind, h, w, p, g):
    """A binary mask: i.i.d. noise, blobs, or one-pixel concentric rings."""
    if kind == "noise":
        return torch.rand((h, w), generator=g, device="cuda") < p
    if kind == "blobs":
        return _smooth(h, w, g)[0] > 0.5
    y = torch.arange(h, device="cuda").reshape(-1, 1)
    x = torch.arange(w, device="cuda").reshape(1, -1)
    d = torch.minimum(torch.minimum(y, x), torch.minimum(h - 1 - y, w - 1 - x)) % 2 == 0
    # (a few gaps join neighbouring rings, so that every seed is another mask)
    return d | (torch.rand((h, w), generator=g, device="cuda") < 0.001)


# ------------------------------------------------------------------ cases --

def listed():
    return [
        # the smallest evaluation: one slice at scanner size, the case-study
        # spec on 16-bit pixels, prepared once and replayed scan after scan
        dict(name="grow-240-u16-replay", kind="spec", spec="grow", h=240, w=240, dtype="u16",
             conn=8, call="replay"),
        # one formula asked once of one resident image, as at a prompt: the
        # whole call counts, planning and launches included
        dict(name="barrier-512-once", kind="spec", spec="barrier", h=512, w=512, dtype="f32",
             conn=8, call="once"),
        # the case study at the largest slice of the paper, 59 Mpx
        dict(name="grow-7680-replay", kind="spec", spec="grow", h=7680, w=7680, dtype="f32",
             conn=8, call="replay"),
        # the stress test: a 2000-node formula over one 2048 x 2048 image,
        # every output wanted
        dict(name="random-2000-2048", kind="random", nodes=2000, dag=0, h=2048, w=2048, conn=8,
             call="replay"),
        # a mid-sized formula on an odd image under 4-adjacency, asked once
        dict(name="random-300-1111x1733-once", kind="random", nodes=300, dag=3, h=1111, w=1733,
             conn=4, call="once"),
        # a sequential formula f(g(...(x))): every operator waits for the one before
        dict(name="chain-500-2048", kind="chain", nodes=500, dag=0, mix="mixed", h=2048, w=2048,
             conn=8, call="replay"),
        # labelling alone: dense noise at 67 Mpx, and odd-sized smooth blobs
        dict(name="label-noise-8192", kind="label", pattern="noise", p=0.5, h=8192, w=8192, conn=8),
        dict(name="label-blobs-3001x2777-c4", kind="label", pattern="blobs", p=0.5, h=3001, w=2777,
             conn=4),
        # a study's worth of 4-channel slices of uneven sizes, one batch,
        # tuned once and replayed
        dict(name="slices-1024", kind="slices", n=1024, median=240, sizes=0, conn=8),
        # a whole scan at once: the segmentation over a 4-channel volume
        dict(name="volume-155x240x240", kind="volume", d=155, h=240, w=240, conn=26),
        # a served mix: queries of 10 to 2000 nodes over resident images of
        # 128 to 2048 pixels a side, planned and run as one new batch
        dict(name="queries-32", kind="queries", n=32, mix_seed=1, conn=8),
        # channel arithmetic with percentiles on a 16-bit two-channel image
        dict(name="terms-1021x1530-u16", kind="terms", h=1021, w=1530, dtype="u16", conn=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("spec", "spec", "random", "random", "chain", "label", "label", "slices",
                       "volume", "queries", "terms"))
    conn = rng.choice((8, 8, 4))
    if kind == "spec":
        return dict(kind=kind, spec=rng.choice(("grow", "barrier")), h=_log_int(rng, 128, 7680),
                    w=_log_int(rng, 128, 7680), dtype=rng.choice(("f32", "u16")), conn=conn,
                    call=rng.choice(("replay", "once")))
    if kind == "random":
        nodes = _log_int(rng, 10, 2000)
        top = min(4096, int(2048 * math.sqrt(2000 / nodes)))
        return dict(kind=kind, nodes=nodes, dag=rng.randrange(1000), h=_log_int(rng, 128, top),
                    w=_log_int(rng, 128, top), conn=conn, call=rng.choice(("replay", "once")))
    if kind == "chain":
        return dict(kind=kind, nodes=_log_int(rng, 10, 500), dag=rng.randrange(1000),
                    mix=rng.choice(sorted(CHAIN_MIXES)), h=_log_int(rng, 128, 2048),
                    w=_log_int(rng, 128, 2048), conn=conn, call=rng.choice(("replay", "once")))
    if kind == "label":
        return dict(kind=kind, pattern=rng.choice(("noise", "noise", "blobs", "rings")),
                    p=rng.uniform(0.3, 0.6), h=_log_int(rng, 256, 8192), w=_log_int(rng, 256, 8192),
                    conn=conn)
    if kind == "slices":
        return dict(kind=kind, n=_log_int(rng, 16, 1024), median=240, sizes=rng.randrange(1, 1000),
                    conn=conn)
    if kind == "volume":
        return dict(kind=kind, d=_log_int(rng, 12, 155), h=rng.randrange(64, 241),
                    w=rng.randrange(64, 241), conn=rng.choice((26, 26, 6)))
    if kind == "queries":
        return dict(kind=kind, n=_log_int(rng, 4, 16), mix_seed=rng.randrange(2, 1000), conn=conn)
    return dict(kind=kind, h=_log_int(rng, 128, 2048), w=_log_int(rng, 128, 2048),
                dtype=rng.choice(("f32", "u16")), conn=conn)


_session = {}


def _open():
    """The program's one context and stream."""
    if not _session:
        _session["ctx"] = vg.Context()
        _session["stream"] = torch.cuda.Stream()
    return _session["ctx"], _session["stream"]


def _words(w):
    """32-pixel words of a packed row."""
    return 4 * ((w + 127) // 128)


def _sides(case):
    """Side lengths of the slices: log-normal around the median, 160 to 512."""
    rng = random.Random(case["sizes"])

    def side():
        return min(512, max(160, round(case["median"] * math.exp(0.25 * rng.gauss(0, 1)))))

    return [(side(), side()) for _ in range(case["n"])]


def _queries(case):
    """(nodes, dag, side) of every query of a mix: sizes log-uniform."""
    rng = random.Random(case["mix_seed"])
    return [(_log_int(rng, 10, 2000), rng.randrange(16), _log_int(rng, 128, 2048))
            for _ in range(case["n"])]


def _spec_text(case):
    if case["spec"] == "barrier":
        return BARRIER if case["dtype"] == "f32" else BARRIER.replace("0.6", "39321").replace("0.3", "19660")
    if case["dtype"] == "f32":
        return GROW.format(hi=0.95, vi=0.86)
    return GROW.format(hi=62258, vi=56360)


def _formula(ctx, case):
    kind = case["kind"]
    if kind == "random":
        return ctx.compile(*_random_dag(case["nodes"], case["dag"]), case["conn"])
    if kind == "chain":
        return ctx.compile(*_chain(case["nodes"], case["dag"], case["mix"]), case["conn"])
    text = {"spec": _spec_text, "terms": lambda c: TERMS}.get(kind, lambda c: SEGMENT)(case)
    return ctx.compile_text(text, case["conn"])


def _image(ctx, case, stream, rng, g):
    h, w = case["h"], case["w"]
    if case["kind"] == "terms":
        x = torch.cat([_upscaled_slice(h, w, rng, g), _upscaled_slice(h, w, rng, g)])
        x = (x + 0.05 * torch.randn(x.shape, generator=g, device="cuda")).clamp(0, 1)
    elif case["kind"] in ("random", "chain"):
        x = _uniform(1, h, w, g)
    else:
        x = _smooth(h, w, g) if case["spec"] == "barrier" else _upscaled_slice(h, w, rng, g)
    if case.get("dtype") == "u16":
        x = _to_u16(x)
    return _resident(ctx.image(x, stream))


def _resident(image):
    image.release_source()
    return image


def _mask_buffer(roots, h, w):
    return torch.empty((roots, h, _words(w)), dtype=torch.int32, device="cuda")


def prepare(case, seed):
    ctx, stream = _open()
    rng, g = random.Random(int(seed)), _generator(seed)
    kind = case["kind"]
    with torch.cuda.stream(stream):
        if kind == "label":
            m = _pattern(case["pattern"], case["h"], case["w"], case["p"], g)
            mask = _resident(ctx.mask(m.to(torch.uint8), stream))
            labels = torch.empty(case["h"] * case["w"], dtype=torch.int32, device="cuda")
            state = dict(do="label", mask=mask, labels=labels, conn=case["conn"])
        elif kind == "slices":
            F = _formula(ctx, case)
            jobs = [(F, [_resident(ctx.image(_phantom(s, rng, g), stream))]) for s in _sides(case)]
            state = _replay(ctx, stream, jobs)
        elif kind == "queries":
            forms, jobs = {}, []
            for nodes, dag, side in _queries(case):
                if (nodes, dag) not in forms:
                    forms[nodes, dag] = ctx.compile(*_random_dag(nodes, dag), case["conn"])
                jobs.append((forms[nodes, dag], [_resident(ctx.image(_uniform(1, side, side, g), stream))]))
            outs = [_mask_buffer(f.info()["n_roots"], im.h, im.w) for f, (im,) in jobs]
            state = dict(do="queries", jobs=jobs, outs=outs)
        elif kind == "volume":
            scan = _phantom((case["d"], case["h"], case["w"]), rng, g).cpu().numpy()
            F, vol = _formula(ctx, case), _resident(ctx.volume(scan, stream))
            stream.synchronize()
            out = _mask_buffer(F.info()["n_roots"], case["d"] * case["h"], case["w"])
            state = dict(do="once", formula=F, images=[vol], out=out)
        else:
            F, im = _formula(ctx, case), _image(ctx, case, stream, rng, g)
            if case.get("call", "once") == "replay":
                state = _replay(ctx, stream, [(F, [im])])
            else:
                out = _mask_buffer(F.info()["n_roots"], case["h"], case["w"])
                state = dict(do="once", formula=F, images=[im], out=out)
    return dict(state, ctx=ctx, stream=stream)


def _replay(ctx, stream, jobs):
    """A prepared batch, its tile shape measured once per formula and size."""
    if not ctx.tile_shape(jobs)["tuned"]:
        ctx.autotune(jobs, stream=stream)
    batch = ctx.batch(jobs, stream)
    results = [batch.result(k) for k in range(len(jobs))]
    if len(jobs) == 1:
        outs = [_mask_buffer(results[0].n_roots, results[0].h, results[0].w)]
    else:
        # one buffer for the masks of all slices, back to back
        words = [r.n_roots * r.h * r.wp for r in results]
        whole = torch.empty(sum(words), dtype=torch.int32, device="cuda")
        outs = list(whole.split(words))
        return dict(do="replay", batch=batch, results=results, outs=outs, whole=whole)
    return dict(do="replay", batch=batch, results=results, outs=outs, whole=outs[0])


def run(state):
    ctx, stream, do = state["ctx"], state["stream"], state["do"]
    if do == "label":
        ctx.ccl(state["mask"], state["labels"], state["conn"], stream)
        return state["labels"]
    if do == "replay":
        state["batch"].run(stream)
        for r, out in zip(state["results"], state["outs"]):
            r.masks_into(out, True, stream)
        return state["whole"]
    if do == "once":
        r = ctx.eval(state["formula"], state["images"], stream)
        r.masks_into(state["out"], True, stream)
        return state["out"]
    for r, out in zip(ctx.eval_batch(state["jobs"], stream), state["outs"]):
        r.masks_into(out, True, stream)
    return state["outs"]


def work(case):
    """Bytes a pass cannot do without: every channel that is read once, every
    output mask or label once.  The arithmetic is bit logic on packed words."""
    kind = case["kind"]
    px = {"u16": 2, "f32": 4}[case.get("dtype", "f32")]

    def masks(roots, h, w):
        return 4 * roots * h * _words(w)

    if kind == "label":
        total = case["h"] * (4 * _words(case["w"]) + 4 * case["w"])
    elif kind == "slices":
        total = sum(4 * 4 * h * w + masks(4, h, w) for h, w in _sides(case))
    elif kind == "volume":
        n = case["d"] * case["h"]
        total = 4 * 4 * n * case["w"] + masks(4, n, case["w"])
    elif kind == "queries":
        total = sum(4 * s * s + masks(len(_random_dag(n, k)[1]), s, s) for n, k, s in _queries(case))
    else:
        roots = {"random": lambda: len(_random_dag(case["nodes"], case["dag"])[1]),
                 "chain": lambda: len(_chain(case["nodes"], case["dag"], case["mix"])[1]),
                 "terms": lambda: 2,
                 "spec": lambda: 2 if case["spec"] == "barrier" else 1}[kind]()
        channels = 2 if kind == "terms" else 1
        total = channels * px * case["h"] * case["w"] + masks(roots, case["h"], case["w"])
    return {"bytes": total, "flops": 0}


def exact(case, seed):
    """Masks and labels are whole numbers: they are right or wrong, not near."""
    return None
