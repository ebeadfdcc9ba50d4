"""The work this framework is timed on, through its public entry points.

Frames follow the repository's generative model (Poisson sky and stars, straight
cosmic-ray tracks, Gaussian read noise, divided by the gain), made on the GPU
from the seed alone. Every clean runs the default method parameters (sigclip
4.5, sigfrac 0.5, objlim 1) unless the case says otherwise.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1008_2192_gb300 import Cleaner, Server, poisson_batch_into, poisson_into
from paper_1008_2192_gb300 import partition

CR_DENSITY = 1500 / 800**2      # cosmic rays per pixel
STAR_DENSITY = 200 / 800**2     # stars per pixel
SIZES = [(800, 800), (1024, 1024), (2048, 4096), (4096, 4096)]  # (w, h) of the mixed batches


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, w=0, h=0, n=1, niter=4, objlim_form=0, graphs=False, autotune=False, parts=0,
             mean=0.0, mixed=False)
    c.update(kw)
    return c


def listed():
    return [
        # one sub-image of the paper's 6 x 6 cut of a 750 x 750 image: the smallest call, launches and latency
        _case("actor_137", "frame", w=137, h=137),
        # one WFPC2 chip, the paper's own frame size
        _case("wfpc2_800", "frame", w=800, h=800),
        # a ragged frame: odd row pitch, no 16-byte row alignment; the article's form of the objlim test
        _case("ragged_1531x1021", "frame", w=1531, h=1021, objlim_form=1),
        # a 2k x 2k detector
        _case("ccd_2048", "frame", w=2048, h=2048),
        # one chip of a two-chip 4k camera, ragged by its overscan columns and rows
        _case("chip_4146x2051", "frame", w=4146, h=2051),
        # a 4k x 4k detector cleaned over and over with one handle, its launches replayed as a graph
        _case("ccd_4096_graph", "frame", w=4096, h=4096, graphs=True),
        # a 1 GiB mosaic in one call: the largest frame
        _case("mosaic_16384", "frame", w=16384, h=16384),
        # the batch workload: 64 uneven frames with their own gains and read noises, tuned and replayed
        _case("batch_64", "batch", n=64, mixed=True, graphs=True, autotune=True),
        # frames in page-locked host memory, through the copy pipeline and back
        _case("host_batch_12", "host", n=12, mixed=True),
        # a burst of frames of mixed sizes through the continuous-batching server
        _case("serve_24", "serve", n=24, mixed=True),
        # the paper's 2-D segmentation of one frame into 6 x 6 sub-images with overlap
        _case("rects_36_of_2048", "rects", w=2048, h=2048, parts=36),
        # the POISSON work function on the paper's 750 x 750 image of mean 24.3
        _case("poisson_750", "poisson", w=750, h=750, mean=24.3),
    ]


def _log_int(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "batch", "host", "serve", "rects", "poisson"])
    form, niter = rng.choice([0, 0, 1]), rng.choice([2, 3, 4, 4, 5])
    if kind == "frame":
        w, h = _log_int(rng, 100, 9000), _log_int(rng, 100, 9000)
        return _case("", kind, w=w, h=h, niter=niter, objlim_form=form, graphs=rng.random() < 0.3)
    if kind in ("batch", "host"):
        w, h = _log_int(rng, 300, 3000), _log_int(rng, 300, 3000)
        return _case("", kind, n=rng.randint(2, 12), w=w, h=h, niter=niter, objlim_form=form,
                     mixed=rng.random() < 0.3)
    if kind == "serve":
        w, h = _log_int(rng, 300, 3000), _log_int(rng, 300, 3000)
        return _case("", kind, n=rng.randint(4, 24), w=w, h=h, niter=niter, mixed=rng.random() < 0.5)
    if kind == "rects":
        return _case("", kind, w=_log_int(rng, 700, 5000), h=_log_int(rng, 700, 5000), niter=niter,
                     objlim_form=form, parts=rng.choice([4, 6, 7, 9, 16, 36]))
    return _case("", kind, w=_log_int(rng, 150, 3000), h=_log_int(rng, 150, 3000), n=rng.choice([1, 1, 4]),
                 mean=round(math.exp(rng.uniform(math.log(2.0), math.log(250.0))), 2))


# ---- inputs ----------------------------------------------------------------------------------------------------

def _sizes(case):
    """(w, h) of the frames: grouped by size, so that frames of a size are one tensor."""
    if case["mixed"]:
        return [SIZES[i * len(SIZES) // case["n"]] for i in range(case["n"])]
    return [(case["w"], case["h"])] * case["n"]


def _groups(case):
    out = []
    for wh in _sizes(case):
        if out and out[-1][0] == wh:
            out[-1][1] += 1
        else:
            out.append([wh, 1])
    return [(wh, k) for wh, k in out]


def _rand(gen, *shape, dtype=torch.float64):
    return torch.rand(*shape, generator=gen, device="cuda", dtype=dtype)


def _frame(out, gen, gain, rn):
    """One synthetic frame in DN into out (h, w)."""
    h, w = out.shape
    sky = 300.0 if w * h >= 4096 * 4096 else 100.0
    nstars, ncr = max(1, round(STAR_DENSITY * w * h)), max(1, round(CR_DENSITY * w * h))
    e = torch.full((h * w,), sky, device="cuda")
    for a in range(0, nstars, 50000):  # pixel-integrated Gaussians, FWHM 1.5-2.5 px, 1e3-1e6 e-
        m = min(50000, nstars - a)
        xc, yc, fw, fl = _rand(gen, m) * w, _rand(gen, m) * h, 1.5 + _rand(gen, m), 10 ** (3 + 3 * _rand(gen, m))
        k = 2.3548200450309493 / (math.sqrt(2.0) * fw)
        o = torch.arange(-7, 8, device="cuda", dtype=torch.float64)
        px, py = xc.floor()[:, None] + o, yc.floor()[:, None] + o
        gx = 0.5 * (torch.erf((px + 1 - xc[:, None]) * k[:, None]) - torch.erf((px - xc[:, None]) * k[:, None]))
        gy = 0.5 * (torch.erf((py + 1 - yc[:, None]) * k[:, None]) - torch.erf((py - yc[:, None]) * k[:, None]))
        v = (fl[:, None, None] * gy[:, :, None] * gx[:, None, :]).float()
        ok = ((py >= 0) & (py < h))[:, :, None] & ((px >= 0) & (px < w))[:, None, :]
        i = (py[:, :, None] * w + px[:, None, :]).long()
        e.index_put_((i[ok],), v[ok], accumulate=True)
    e = torch.poisson(e, generator=gen)
    e += rn * torch.randn(h * w, generator=gen, device="cuda")
    # tracks of 1-10 px sampled every quarter pixel (a fifth are single hits), 1e2-1e4 e- on each pixel touched
    xs, ys, th = _rand(gen, ncr) * w, _rand(gen, ncr) * h, _rand(gen, ncr) * math.pi
    single, ln, amp = _rand(gen, ncr) < 0.2, 1 + 9 * _rand(gen, ncr), 10 ** (2 + 2 * _rand(gen, ncr))
    t = torch.arange(0, 41, device="cuda", dtype=torch.float64) * 0.25
    px = (xs[:, None] + t * torch.cos(th)[:, None]).floor()
    py = (ys[:, None] + t * torch.sin(th)[:, None]).floor()
    on = (t <= torch.where(single, 0.0, ln)[:, None]) & (px >= 0) & (px < w) & (py >= 0) & (py < h)
    i = (py * w + px).long()
    on[:, 1:] &= i[:, 1:] != i[:, :-1]  # a pixel once per track
    e.index_put_((i[on],), amp.float()[:, None].expand(i.shape)[on], accumulate=True)
    torch.div(e.view(h, w), gain, out=out)


def _inputs(case, seed):
    """The case's input frames, one tensor per size, with their gains and read noises."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 1000003 + 17)
    rng = np.random.default_rng([int(seed), 11])
    stacks, gains, rns = [], [], []
    many = case["n"] > 1 or case["kind"] in ("batch", "host", "serve")
    for (w, h), k in _groups(case):
        s = torch.empty((k, h, w), device="cuda")
        for j in range(k):
            g, r = (float(np.float32(rng.uniform(1, 7))), float(np.float32(rng.uniform(3, 10)))) if many else (7.0, 5.0)
            _frame(s[j], gen, g, r)
            gains.append(g)
            rns.append(r)
        stacks.append(s)
    return stacks, gains, rns


def _means(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 1000003 + 29)
    m = torch.rand(case["n"], case["h"], case["w"], generator=gen, device="cuda")
    return [(case["mean"] * (0.9 + 0.2 * m)).contiguous()], [int(seed) * 7919 + i for i in range(case["n"])]


def _options(case):
    return dict(gain=7.0, readnoise=5.0, niter=case["niter"], objlim_form=case["objlim_form"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        imgs, seeds = _means(case, seed)
        return dict(kind=kind, imgs=list(imgs[0]), out=torch.empty_like(imgs[0]), seeds=seeds)
    stacks, gains, rns = _inputs(case, seed)
    st = dict(kind=kind, gains=gains, rns=rns)
    if kind == "host":
        stacks = [s.cpu().pin_memory() for s in stacks]
        st["outs"] = [torch.empty(s.shape, pin_memory=True) for s in stacks]
        st["masks"] = [torch.empty(s.shape, dtype=torch.uint8, pin_memory=True) for s in stacks]
    else:
        st["outs"] = [torch.empty_like(s) for s in stacks]
        st["masks"] = [torch.empty(s.shape, dtype=torch.uint8, device="cuda") for s in stacks]
    st["f_img"] = [f for s in stacks for f in s]
    st["f_out"] = [f for s in st["outs"] for f in s]
    st["f_mask"] = [f for s in st["masks"] for f in s]
    if kind == "serve":
        st["server"] = Server(**_options(case))
    else:
        st["cleaner"] = Cleaner(**_options(case), use_graphs=case["graphs"], autotune=case["autotune"])
    if kind == "rects":
        st["rects"] = partition.plan(case["w"], case["h"], case["parts"], 8 * case["niter"])[2]
    return st


def run(state):
    kind = state["kind"]
    if kind == "poisson":
        if len(state["imgs"]) == 1:
            poisson_into(state["imgs"][0], state["out"][0], state["seeds"][0])
        else:
            poisson_batch_into(state["imgs"], list(state["out"]), state["seeds"])
        return [state["out"]]
    img, out, mask = state["f_img"], state["f_out"], state["f_mask"]
    if kind == "frame":
        state["cleaner"].clean_into(img[0], out[0], mask[0])
    elif kind == "rects":
        state["cleaner"].clean_rects_into(img[0], state["rects"], out[0], mask[0])
    elif kind == "batch":
        state["cleaner"].clean_batch_into(img, out, mask, state["gains"], state["rns"])
    elif kind == "host":
        state["cleaner"].clean_batch_host_into(img, out, mask, state["gains"], state["rns"])
    else:
        srv, left = state["server"], len(img)
        for i in range(len(img)):
            while not srv.submit(img[i], out[i], mask[i], i, state["gains"][i], state["rns"][i]):
                left -= len(srv.poll(block_ms=100))
        while left:
            left -= len(srv.poll(block_ms=1000))
    return dict(clean=state["outs"], mask=state["masks"])


def work(case):
    px = sum(w * h for w, h in _sizes(case))
    if case["kind"] == "poisson":  # mean in, deviate out; one product per factor drawn
        return {"bytes": 8.0 * px, "flops": px * (case["mean"] + 1)}
    # image in, cleaned image and mask out; the test of every pixel against its threshold once (35 operations)
    return {"bytes": 9.0 * px, "flops": 35.0 * px}


# ---- the same in 64 bits, from the definitions ---------------------------------------------------------------------

def _network(n):
    """Compare-exchange pairs that sort n values (Batcher's merge exchange, Knuth's Algorithm M)."""
    t = max(1, math.ceil(math.log2(n)))
    p, pairs = 1 << (t - 1), []
    while p > 0:
        q, r, d = 1 << (t - 1), 0, p
        while True:
            pairs += [(i, i + d) for i in range(n - d) if (i & p) == r]
            if q == p:
                break
            d, q, r = q - p, q >> 1, p
        p >>= 1
    return pairs


def _windows(a, r):
    """The (2r+1)^2 shifted copies of a, coordinates clamped to the frame."""
    h, w = a.shape
    y, x = torch.arange(h, device=a.device), torch.arange(w, device=a.device)
    rows = [a[(y + d).clamp(0, h - 1)] for d in range(-r, r + 1)]
    return [q[:, (x + d).clamp(0, w - 1)] for q in rows for d in range(-r, r + 1)]


def _median(a, r):
    v = _windows(a, r)
    for i, j in _network(len(v)):
        v[i], v[j] = torch.minimum(v[i], v[j]), torch.maximum(v[i], v[j])
    return v[len(v) // 2]


def _grow(m):
    return torch.nn.functional.max_pool2d(m[None, None].float(), 3, 1, 1)[0, 0] > 0


def _clean64(img, gain, rn, niter, form, sigclip=4.5, sigfrac=0.5, objlim=1.0):
    J = img.double()
    h, w = J.shape
    M = torch.zeros(h, w, dtype=torch.bool, device=J.device)
    for _ in range(niter):
        c = _windows(J, 1)
        cl = lambda t: t.clamp(min=0)  # noqa: E731
        up, le, ri, dn = c[1], c[3], c[5], c[7]
        lp = (cl(2 * J - up - le) + cl(2 * J - up - ri) + cl(2 * J - dn - le) + cl(2 * J - dn - ri)) / 4
        m5 = _median(J, 2)
        m5 = torch.where(m5 <= 0, 1e-4, m5)
        N = torch.sqrt(gain * m5 + rn * rn) / gain
        S = lp / (2 * N)
        Sp = S - _median(S, 2)
        m3 = _median(J, 1)
        F = ((m3 - _median(m3, 3)) / N).clamp(min=0.01)
        hit = (Sp > sigclip) & ((2 * S if form else Sp) / F > objlim)
        g1 = _grow(hit) & (Sp > sigclip)
        M |= _grow(g1) & (Sp > sigfrac * sigclip)
        y, x = M.nonzero(as_tuple=True)
        o = torch.arange(-2, 3, device=J.device)
        yy = (y[:, None, None] + o[:, None]).clamp(0, h - 1).expand(-1, 5, 5).reshape(-1, 25)
        xx = (x[:, None, None] + o).clamp(0, w - 1).expand(-1, 5, 5).reshape(-1, 25)
        v, f = J[yy, xx], M[yy, xx]
        v = v.masked_fill(f, math.inf).sort(dim=1).values
        k = 25 - f.sum(1)
        val = v.gather(1, ((k + 1) // 2 - 1).clamp(min=0)[:, None])[:, 0]
        J = J.clone()
        J[y, x] = torch.where(k > 0, val, m5[y, x])
    return J


def _banded64(img, gain, rn, niter, form):
    """_clean64 by bands of rows with the context that leaves their interiors exact (8 rows an iteration)."""
    h, w = img.shape
    step, ctx, out = max(64, (1 << 24) // w), 8 * niter, []
    for a in range(0, h, step):
        b = min(h, a + step)
        lo, hi = max(0, a - ctx), min(h, b + ctx)
        out.append(_clean64(img[lo:hi], gain, rn, niter, form)[a - lo:b - lo].to(torch.float64))
    return torch.cat(out)


def _poisson64(mu, seed):
    """Knuth's multiplicative method on SplitMix64 streams keyed by the pixel."""
    g, one = np.uint64(0x9E3779B97F4A7C15), np.uint64(1)

    def mix(z):
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return z ^ (z >> np.uint64(31))

    with np.errstate(over="ignore"):
        m = mu.double().cpu().numpy().reshape(-1)
        lim = np.exp(-np.minimum(m, 700.0))
        key = mix(np.uint64(seed & (2**64 - 1)) + (np.arange(m.size, dtype=np.uint64) + one) * g)
        k, q, live, j = np.zeros(m.size), np.ones(m.size), np.flatnonzero(m > 0), 0
        while live.size and j <= 4096:
            j += 1
            u = (mix(key[live] + np.uint64(j) * g) >> np.uint64(11)) * 2.0**-53
            q[live] *= u
            live = live[q[live] >= lim[live]]
            k[live] = j
    return torch.from_numpy(np.minimum(k, 4096)).reshape(mu.shape)


def exact(case, seed):
    px = sum(w * h for w, h in _sizes(case))
    if case["kind"] == "poisson":
        if px * case["mean"] > 5e8:
            return None
        imgs, seeds = _means(case, seed)
        return [torch.stack([_poisson64(m, s) for m, s in zip(imgs[0], seeds)])]
    stacks, gains, rns = _inputs(case, seed)
    clean, i = [], 0
    for s in stacks:
        res = torch.empty(s.shape, dtype=torch.float64, device="cuda")
        for j in range(s.shape[0]):
            res[j] = _banded64(s[j], gains[i], rns[i], case["niter"], case["objlim_form"])
            i += 1
        clean.append(res)
    return dict(clean=clean, mask=[None] * len(clean))
