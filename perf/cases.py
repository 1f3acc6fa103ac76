"""The work a user of this library has it do, as measurable cases.

Every case goes through the package's public entry points: one-shot Vegas
calls, device-resident integrals, single sampling passes (DoSample), batches,
the request server, user integrands on materialised samples, and Suave.
Integrand parameters follow the repository's workloads: `a` drawn from U(0,1)
and scaled to a given difficulty (genz8d4c: sum 8), or 1/2 + U(0,1) (the
batch and the server); `u` from U(0,1).

What `run` hands back is what the call computed.  The FP32 path evaluates
points and integrands in binary32, so its numbers are handed on as float32;
the FP64 path's stay float64.  The chi-square probability is returned on the
FP64 path only: on the FP32 path it is a steep function of differences
between iteration results that lie below that path's own accuracy (Sobol
points make those differences far smaller than the error estimate), and the
iteration results themselves are returned where the entry point gives them.

`exact` is the same Vegas (Sobol points of the same 23 or 52 bits, the same
grid refinement and combination) in plain torch and numpy at 64 bits.
"""
import math

import numpy as np
import torch

import paper_1408_6373_gb300 as cg
from paper_1408_6373_gb300.workloads import fp32_corner_peak

OSC, PROD, CORNER, GAUSS, C0, DISC = range(6)


# ------------------------------------------------------------------ cases
def listed():
    return [
        # The smallest call: a 3-D peak in double precision, ten iterations
        # of 1e4 points (the repository's gaussian3d configuration), as a
        # program that integrates inside another loop makes it.
        dict(name="vegas_gaussian3d_fp64", kind="vegas", ndim=3, fams="3", nbins=50, nstart=10000, ninc=0,
             iters=10, fp64=True, gen="sobol", hard=15.0),
        # An ordinary call with every default: two components in six
        # dimensions, 64 bins, growing iterations of ragged size.
        dict(name="vegas_ordinary", kind="vegas", ndim=6, fams="13", nbins=64, nstart=100003, ninc=50001,
             iters=8, fp64=False, gen="sobol", hard=9.0),
        # The headline integral (genz8d4c): four components, 20 iterations of
        # 1e7 points on a handle a program keeps, specialised at run time.
        dict(name="integral_genz8d4c_jit", kind="integral", ndim=8, fams="0123", nbins=128, nstart=10000000,
             ninc=0, iters=20, jit=True, gen="sobol", hard=8.0),
        # One DoSample pass as a program with its own Vegas driver makes it:
        # the general kernel, an adapted grid, a start and a count that are
        # not multiples of anything.
        dict(name="pass_genz8d4c", kind="sample", ndim=8, fams="0123", nbins=128, start=30000001, n=9999991,
             fp64=False, gen="sobol", hard=8.0),
        # The same pass in double precision, for accuracy below 1e-7.
        dict(name="pass_fp64", kind="sample", ndim=8, fams="0123", nbins=128, start=5000011, n=1000003,
             fp64=True, gen="sobol", hard=8.0),
        # Independent points (error bars without net structure): pseudo-random
        # sampling, five dimensions, 100 bins.
        dict(name="integral_pseudo", kind="integral", ndim=5, fams="34", nbins=100, nstart=2000000, ninc=0,
             iters=5, jit=False, gen="pseudo", hard=7.0),
        # Many integrals of a parameter scan at once (the batch4096 mix, 512
        # of them, 1e4 to 1e6 points an iteration).
        dict(name="batch_512", kind="batch", count=512, dmin=2, dmax=16, nbins=64, nmin=10000, nmax=1000000,
             iters=5),
        # A burst of requests to the server: 2 to 16 dimensions, 1 to 4
        # components, accuracy goals of 1e-5 to 1e-3.
        dict(name="serve_burst_96", kind="serve", count=96, dmin=2, dmax=16, nbins=64, maxeval=10000000),
        # The user's own integrand on materialised samples, dimension-major,
        # one tile per iteration of 1e7 points (the library's specialised
        # device integrand stands for the user's).
        dict(name="callback_genz8d4c", kind="callback", ndim=8, fams="0123", nbins=128, nstart=10000000, ninc=0,
             iters=4, nvec=10000000, fp64=False, aos=False, jit=True, hard=8.0),
        # The paper's point-major contract x[nvec][ndim], tiles of at most
        # 1e6 points with a ragged last one.
        dict(name="callback_point_major", kind="callback", ndim=5, fams="13", nbins=64, nstart=2500001, ninc=0,
             iters=4, nvec=1000000, fp64=False, aos=True, jit=False, hard=8.0),
        # Suave on a peaked 6-D Gaussian.
        dict(name="suave_6d", kind="suave", ndim=6, fams="3", nbins=16, nnew=65536, width=16, maxeval=60000000,
             max_regions=512, hard=18.0),
        # A single large integral in 30 dimensions with 256 bins (large30d,
        # fewer and smaller iterations).
        dict(name="integral_30d", kind="integral", ndim=30, fams="4", nbins=256, nstart=50000000, ninc=0,
             iters=3, jit=False, gen="sobol", hard=15.0),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def families(k):
        return "".join(str(rng.choice([OSC, PROD, CORNER, GAUSS, C0])) for _ in range(k))

    kind = rng.choice(["vegas", "vegas", "vegas", "integral", "sample", "sample", "batch", "serve", "callback",
                       "suave"])
    nbins = rng.choice([32, 50, 64, 64, 100, 128, 128, 256, rng.randint(20, 256)])
    gen = rng.choice(["sobol", "sobol", "scramble", "pseudo"])
    most = 1000000 if gen == "pseudo" else 10000000
    if kind == "vegas":
        fp64 = rng.random() < 0.3
        return dict(kind=kind, ndim=rng.randint(2, 12), fams=families(rng.randint(1, 4)), nbins=nbins,
                    nstart=logint(10000, 200000 if fp64 else most // 2), ninc=rng.choice([0, logint(1000, 100000)]),
                    iters=rng.randint(2, 12), fp64=fp64, gen=gen, hard=rng.uniform(4.0, 9.0))
    if kind == "integral":
        ndim = rng.choice([rng.randint(2, 12), rng.randint(13, 32)])
        return dict(kind=kind, ndim=ndim, fams=families(rng.randint(1, 4)) if ndim <= 12 else rng.choice("034"),
                    nbins=nbins, nstart=logint(100000, most), ninc=0, iters=rng.randint(2, 8),
                    jit=rng.random() < 0.3, gen=gen, hard=rng.uniform(4.0, 9.0))
    if kind == "sample":
        fp64 = rng.random() < 0.4
        return dict(kind=kind, ndim=rng.randint(2, 16), fams=families(rng.randint(1, 4)), nbins=nbins,
                    start=logint(1, 100000000), n=logint(10000, 1000000 if fp64 else most), fp64=fp64,
                    gen=gen, hard=rng.uniform(4.0, 9.0))
    if kind == "batch":
        return dict(kind=kind, count=logint(8, 512), dmin=2, dmax=rng.randint(3, 16),
                    nbins=rng.choice([32, 50, 64, 128]), nmin=10000, nmax=logint(20000, 1000000),
                    iters=rng.randint(2, 5))
    if kind == "serve":
        return dict(kind=kind, count=logint(1, 96), dmin=2, dmax=rng.randint(3, 16), nbins=rng.choice([50, 64, 128]),
                    maxeval=logint(500000, 10000000))
    if kind == "callback":
        fp64, aos = rng.random() < 0.2, rng.random() < 0.4
        return dict(kind=kind, ndim=rng.randint(2, 10), fams=families(rng.randint(1, 4)), nbins=nbins,
                    nstart=logint(50000, 400000 if fp64 else 5000000), ninc=0, iters=rng.randint(2, 5),
                    nvec=logint(50000, 5000000), fp64=fp64, aos=aos, jit=False, hard=rng.uniform(4.0, 9.0))
    return dict(kind=kind, ndim=rng.randint(2, 8), fams=rng.choice("134"), nbins=rng.choice([8, 16, 32]),
                nnew=logint(4096, 65536), width=rng.choice([1, 4, 16]), maxeval=logint(1000000, 60000000),
                max_regions=256, hard=rng.uniform(6.0, 18.0))


# ------------------------------------------------------------------ inputs
def _parameters(rng, ndim, fams, hard):
    """a[c, d] (scaled to sum `hard` per component), u[c, d]."""
    a, u = rng.random((len(fams), ndim)), rng.random((len(fams), ndim))
    a = 0.05 + a
    a *= hard / a.sum(axis=1, keepdims=True)
    for c, f in enumerate(fams):
        if f == CORNER:
            a[c] = fp32_corner_peak(a[c])
    return a, u


def _many(case, seed):
    """The integrands of a batch or of a burst of requests."""
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(case["count"]):
        ndim = int(rng.integers(case["dmin"], case["dmax"] + 1))
        ncomp = int(rng.integers(1, 5)) if case["kind"] == "serve" else 1
        # (the discontinuous family in few dimensions only, where its estimate
        # does not hang on single points, and not as the first of several
        # components: a grid that follows it leaves the others unsampled)
        fams = [int(rng.integers(0, 5 if ndim > 6 or (c == 0 and ncomp > 1) else 6)) for c in range(ncomp)]
        a, u = 0.5 + rng.random((ncomp, ndim)), rng.random((ncomp, ndim))
        for c, f in enumerate(fams):
            if f == CORNER:
                a[c] = fp32_corner_peak(a[c])
        p = dict(ndim=ndim, fams=fams, a=a, u=u)
        if case["kind"] == "serve":
            p["epsrel"] = float(10.0 ** rng.uniform(-5, -3))
        else:
            p["n"] = int(round(math.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"])))))
        out.append(p)
    return out


def _one(case, seed):
    fams = [int(c) for c in case["fams"]]
    rng = np.random.default_rng(seed)
    a, u = _parameters(rng, case["ndim"], fams, case["hard"])
    edges = None
    if case["kind"] == "sample":
        # an adapted grid: bins that shrink towards a point of every axis
        N = case["nbins"]
        t = np.arange(N + 1) / N
        edges = np.empty((case["ndim"], N + 1))
        for d in range(case["ndim"]):
            amp, phase = rng.uniform(0.3, 0.8), rng.uniform(0, 2 * math.pi)
            e = t + amp / (2 * math.pi) * (np.sin(2 * math.pi * t + phase) - math.sin(phase))
            e[0], e[-1] = 0.0, 1.0
            edges[d] = e
    return dict(ndim=case["ndim"], fams=fams, a=a, u=u, edges=edges)


def _maxeval(nstart, ninc, iters):
    return iters * nstart + ninc * (iters * (iters - 1) // 2)


def _flags(case):
    f = cg.FP64 if case.get("fp64") else 0
    f |= cg.JIT if case.get("jit") and case["kind"] != "callback" else 0
    f |= cg.AOS if case.get("aos") else 0
    return f | {"sobol": 0, "scramble": cg.SCRAMBLE, "pseudo": cg.PSEUDO}[case.get("gen", "sobol")]


_CONTEXT = []


def _context():
    """The library handle a program creates once and keeps."""
    if not _CONTEXT:
        _CONTEXT.append(cg.Context(0))
    return _CONTEXT[0]


def prepare(case, seed):
    ctx = _context()
    s = dict(case=case, ctx=ctx, seed=int(seed) & 0x7fffffff)
    kind = case["kind"]
    if kind in ("batch", "serve"):
        s["specs"] = []
        for p in _many(case, seed):
            g = cg.genz(p["ndim"], p["fams"], p["a"], p["u"])
            if kind == "batch":
                sp = cg.spec(g, nbins=case["nbins"], nstart=p["n"], maxeval=case["iters"] * p["n"])
            else:
                sp = cg.spec(g, nbins=case["nbins"], nstart=10000, nincrease=50000, maxeval=case["maxeval"],
                             epsrel=p["epsrel"])
            s["specs"].append(sp)
        if kind == "batch":
            s["batch"] = ctx.batch(s["specs"])
        else:
            s["server"] = ctx.server()
        return s
    p = _one(case, seed)
    s["g"] = cg.genz(p["ndim"], p["fams"], p["a"], p["u"])
    if kind == "integral":
        s["integral"] = ctx.integral(cg.spec(
            s["g"], nbins=case["nbins"], flags=_flags(case), nstart=case["nstart"], nincrease=case["ninc"],
            maxeval=_maxeval(case["nstart"], case["ninc"], case["iters"]), seed=s["seed"]))
    elif kind == "sample":
        s["edges"] = torch.from_numpy(p["edges"]).cuda()
        nc = len(p["fams"])
        s["sums"] = torch.empty(2 * nc + case["ndim"] * case["nbins"], dtype=torch.float64, device="cuda")
    elif kind == "callback":
        s["userdata"] = cg.GenzCallbackData(s["g"], _flags(case) | (cg.JIT if case["jit"] else 0))
    return s


# ------------------------------------------------------------------ the work
def _hand_on(fp64, **arrays):
    return {k: np.asarray(v, dtype=np.float64 if fp64 else np.float32) for k, v in arrays.items()}


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "vegas":
        r = ctx.vegas(s["g"], flags=_flags(case), seed=s["seed"], nbins=case["nbins"], nstart=case["nstart"],
                      nincrease=case["ninc"], maxeval=_maxeval(case["nstart"], case["ninc"], case["iters"]))
        out = _hand_on(case["fp64"], integral=r.integral, error=r.error)
        if case["fp64"]:
            out["prob"] = r.prob
        return dict(out, neval=r.neval, fail=r.fail)
    if kind == "integral":
        I = s["integral"]
        I.reset()
        I.run()
        r = I.result()
        nc = len(case["fams"])
        it_I, it_var = I.log(case["iters"])
        out = _hand_on(False, integral=r.integral[:nc], error=r.error[:nc], iterations=it_I, variances=it_var,
                       grid=I.grid())
        return dict(out, neval=r.neval, fail=r.fail)
    if kind == "sample":
        nc, sums = len(case["fams"]), s["sums"]
        sums.zero_()
        S1, S2, H = sums[:nc], sums[nc:2 * nc], sums[2 * nc:]
        ctx.sample(s["g"], case["nbins"], s["edges"], case["start"], case["n"], _flags(case), S1, S2, H,
                   seed=s["seed"])
        if not case["fp64"]:
            sums = sums.to(torch.float32)
        return dict(S1=sums[:nc], S2=sums[nc:2 * nc], H=sums[2 * nc:])
    if kind in ("batch", "serve"):
        if kind == "batch":
            s["batch"].run()
            res = s["batch"].results()
        else:
            ids = [s["server"].submit(sp) for sp in s["specs"]]
            res = [s["server"].wait(i) for i in ids]
        nc = max(sp.g.ncomp for sp in s["specs"])
        out = _hand_on(False, integral=[r.integral[:nc] for r in res], error=[r.error[:nc] for r in res])
        return dict(out, neval=np.array([r.neval for r in res]), fail=np.array([r.fail for r in res]))
    if kind == "callback":
        r = ctx.vegas_cb(cg.builtin_integrand(), case["ndim"], len(case["fams"]), userdata=s["userdata"],
                         nvec=case["nvec"], flags=_flags(case), nbins=case["nbins"], nstart=case["nstart"],
                         nincrease=case["ninc"], maxeval=_maxeval(case["nstart"], case["ninc"], case["iters"]))
        out = _hand_on(case["fp64"], integral=r.integral, error=r.error)
        return dict(out, neval=r.neval, fail=r.fail)
    r = ctx.suave(s["g"], nbins=case["nbins"], maxeval=case["maxeval"], nnew=case["nnew"], width=case["width"],
                  max_regions=case["max_regions"])
    out = _hand_on(False, integral=r.integral, error=r.error, boxes=r.boxes)
    return dict(out, nregions=r.nregions, neval=r.neval, fail=r.fail)


# ------------------------------------------------------------------ what it cannot do without
def _flops_per_sample(ndim, fams):
    per = {OSC: 2 * ndim + 3, PROD: 4 * ndim + 1, CORNER: 2 * ndim + 6, GAUSS: 4 * ndim + 1, C0: 3 * ndim + 1,
           DISC: 2 * ndim + 3}
    # map, integrand, J f and its sums, histogram
    return 3 * ndim + sum(per[f] + 10 for f in fams) + ndim + 1


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        ndim = 0.5 * (case["dmin"] + case["dmax"])
        ncomp = 1 if kind == "batch" else 2.5
        if kind == "batch":
            mean = (case["nmax"] - case["nmin"]) / math.log(case["nmax"] / case["nmin"])
            n = case["count"] * case["iters"] * mean
        else:
            n = case["count"] * 0.5 * case["maxeval"]
        flops = n * (3 * ndim + ncomp * (3 * ndim + 14) + ndim + 1)
        return dict(bytes=case["count"] * (2 * ncomp * ndim + 10) * 8.0, flops=float(flops))
    fams = [int(c) for c in case["fams"]]
    ndim, nc = case["ndim"], len(fams)
    grid = 8.0 * ndim * (case["nbins"] + 1)
    if kind == "sample":
        n, nbytes = case["n"], 2 * grid + 16 * nc
    elif kind == "suave":
        n, nbytes = case["maxeval"], 16.0 * ndim * case["max_regions"]
    else:
        n, nbytes = _maxeval(case["nstart"], case["ninc"], case["iters"]), grid + 64 * nc
    if kind == "callback":
        # every point written and read, every value written and read
        nbytes += 2.0 * n * (ndim + nc) * (8 if case["fp64"] else 4)
    return dict(bytes=float(nbytes), flops=float(n) * _flops_per_sample(ndim, fams))


# ------------------------------------------------------------------ the same in 64 bits
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


_TABLES = {}


def _sobol_tables(ndim):
    """XOR of the direction words (30 bits) over the set bits of every
    15-bit value: low and high halves of a Gray-code index."""
    if ndim not in _TABLES:
        v = torch.quasirandom.SobolEngine(ndim).sobolstate.to(torch.int64)
        halves = []
        for h in range(2):
            t = torch.zeros((ndim, 1), dtype=torch.int64)
            for k in range(15):
                t = torch.cat([t, t ^ v[:, 15 * h + k, None]], dim=1)
            halves.append(t.to(_device()))
        _TABLES[ndim] = halves
    return _TABLES[ndim]


def _philox(seed, words, start, n):
    """Philox4x64-10 blocks of counters (start.., *words) under key (seed, 0)
    (numpy advances the counter before each block)."""
    g = np.random.Philox(counter=np.array([start - 1, *words], dtype=np.uint64), key=np.array([seed, 0], dtype=np.uint64))
    return g.random_raw(4 * n).reshape(n, 4)


def _coordinates(ndim, start, n, bits, gen, seed):
    """int64 [ndim, n]: the top `bits` bits of every point's words."""
    if gen == "pseudo":
        cols = [(_philox(seed, (k, 0, 0), start, n) >> np.uint64(64 - bits)).astype(np.int64)
                for k in range((ndim + 3) // 4)]
        return torch.from_numpy(np.ascontiguousarray(np.concatenate(cols, axis=1)[:, :ndim].T)).to(_device())
    lo, hi = _sobol_tables(ndim)
    i = torch.arange(start, start + n, dtype=torch.int64, device=_device())
    g = i ^ (i >> 1)
    x = lo[:, g & 32767] ^ hi[:, g >> 15]  # (indices below 2^30: 30 bits)
    y = x >> (30 - bits) if bits <= 30 else x << (bits - 30)
    if gen == "scramble":
        for d in range(ndim):
            # (counter (0, d/4, 1, 0): the block before it is all-ones with a borrow)
            g4 = np.random.Philox(counter=np.array([2 ** 64 - 1, d // 4 - 1, 1, 0] if d >= 4 else
                                                   [2 ** 64 - 1, 2 ** 64 - 1, 0, 0], dtype=np.uint64),
                                  key=np.array([seed, 0], dtype=np.uint64))
            y[d] ^= int(g4.random_raw(4)[d % 4]) >> (64 - bits)
    return y


def _integrand(fam, a, u, x):
    a, u = a[:, None], u[:, None]
    ndim = x.shape[0]
    if fam == OSC:
        return torch.cos(2 * math.pi * u[0] + (a * x).sum(0))
    if fam == PROD:
        return 1.0 / (a ** -2 + (x - u) ** 2).prod(0)
    if fam == CORNER:
        return (1.0 + (a * x).sum(0)) ** -(ndim + 1.0)
    if fam == GAUSS:
        return torch.exp(-((a * (x - u)) ** 2).sum(0))
    if fam == C0:
        return torch.exp(-(a * (x - u).abs()).sum(0))
    out = (x[0] > u[0]) | (x[1] > u[1]) if ndim > 1 else x[0] > u[0]
    return torch.where(out, torch.zeros_like(x[0]), torch.exp((a * x).sum(0)))


def _pass64(p, edges, start, n, bits, gen="sobol", seed=0):
    """S1[c], S2[c], H[d, k] of one sampling pass, numpy."""
    dev, ndim, N = _device(), p["ndim"], edges.shape[1] - 1
    e = torch.from_numpy(edges).to(dev)
    w = e[:, 1:] - e[:, :-1]
    a, u = (torch.from_numpy(np.asarray(p[k])).to(dev) for k in "au")
    nc = len(p["fams"])
    S1 = torch.zeros(nc, dtype=torch.float64, device=dev)
    S2, H = torch.zeros_like(S1), torch.zeros(ndim * N, dtype=torch.float64, device=dev)
    row = torch.arange(ndim, device=dev)[:, None] * N
    step = max(1 << 15, (1 << 24) // ndim)
    for at in range(0, n, step):
        m = min(step, n - at)
        t = _coordinates(ndim, start + at, m, bits, gen, seed)
        t.mul_(N)  # (60 bits at most)
        k = t >> bits
        frac = (t & ((1 << bits) - 1)).to(torch.float64) * 2.0 ** -bits
        slot = k + row
        ww = w.reshape(-1)[slot]
        x = e[:, :-1].reshape(-1)[slot] + ww * frac
        J = (ww * N).prod(0)
        for c, f in enumerate(p["fams"]):
            v = J * _integrand(f, a[c], u[c], x)
            S1[c] += v.sum()
            S2[c] += (v * v).sum()
            if c == 0:
                h = v * v
        H += torch.bincount(slot.reshape(-1), weights=h.expand(ndim, m).reshape(-1), minlength=ndim * N)
    return S1.cpu().numpy(), S2.cpu().numpy(), H.reshape(ndim, N).cpu().numpy()


def _refine64(H, edges):
    """Lepage's refinement, exponent 1.5, one axis a row; the new edges."""
    out = edges.copy()
    for d in range(H.shape[0]):
        h, e = H[d], edges[d]
        N = len(h)
        if not np.all(np.isfinite(h)) or not np.any(h):
            continue
        s = np.empty(N)
        s[1:-1] = (h[:-2] + h[1:-1] + h[2:]) / 3.0
        s[0], s[-1] = (h[0] + h[1]) / 2.0, (h[-2] + h[-1]) / 2.0
        x = s / s.sum()
        r = np.zeros(N)
        ok = (x > 0) & (x < 1)
        r[ok] = ((x[ok] - 1.0) / np.log(x[ok])) ** 1.5
        r[x >= 1] = 1.0
        r /= r.max()
        C = np.concatenate([[0.0], np.cumsum(r)])
        t = np.arange(1, N) * (C[-1] / N)
        j = np.clip(np.searchsorted(C, t, side="right") - 1, 0, N - 1)
        out[d, 1:N] = e[j] + (e[j + 1] - e[j]) * ((t - C[j]) / r[j])
    return out


def _vegas64(p, nbins, bits, nstart, ninc, maxeval, gen="sobol", seed=0, epsrel=0.0):
    ndim, nc = p["ndim"], len(p["fams"])
    edges = np.tile(np.arange(nbins + 1) / nbins, (ndim, 1))
    its, vrs, neval, start, n, fail = [], [], 0, 1, nstart, 1
    while True:
        S1, S2, H = _pass64(p, edges, start, n, bits, gen, seed)
        I = S1 / n
        its.append(I)
        vrs.append((S2 / n - I * I) / (n - 1))
        edges = _refine64(H, edges)
        neval, start = neval + n, start + n
        I, V = np.array(its), np.array(vrs)
        flat = np.any(V <= 0, axis=0)
        W = 1.0 / np.where(V > 0, V, 1.0)
        mean = np.where(flat, I.mean(0), (W * I).sum(0) / W.sum(0))
        err = np.where(flat, 0.0, 1.0 / np.sqrt(W.sum(0)))
        if np.all(err <= epsrel * np.abs(mean)):
            fail = 0
            break
        n = nstart + len(its) * ninc
        if neval + n > maxeval:
            break
    chi2 = np.where(flat, 0.0, (W * (I - mean) ** 2).sum(0))
    half = torch.full((nc,), 0.5 * (len(its) - 1), dtype=torch.float64)
    prob = torch.special.gammainc(half, torch.from_numpy(0.5 * chi2)).numpy() if len(its) > 1 else np.zeros(nc)
    return dict(integral=mean, error=err, prob=prob, iterations=I, variances=V, grid=edges, neval=neval, fail=fail)


def _suave64(case, p):
    ndim, N, nnew = p["ndim"], case["nbins"], case["nnew"]
    state = dict(next=1, done=0)

    def sample(edges):
        S1, S2, H = _pass64(p, edges, state["next"], nnew, 23)
        state["next"] += nnew
        state["done"] += nnew
        I = S1 / nnew
        return I, np.maximum((S2 / nnew - I * I) / (nnew - 1), 0.0), H

    def adapt(edges):
        I, V, H = sample(edges)
        new = _refine64(H, edges)
        w = np.diff(new, axis=1)
        fl = np.sqrt((np.log(w / w.mean(axis=1, keepdims=True)) ** 2).mean(axis=1))
        return [new, I, V, fl]

    R = [adapt(np.tile(np.arange(N + 1) / N, (ndim, 1)))]
    while True:
        if all(math.sqrt(sum(r[2][c] for r in R)) <= 0.0 for c in range(len(p["fams"]))):
            break
        order = sorted((k for k in range(len(R)) if R[k][2][0] > 0), key=lambda k: (-R[k][2][0], k))
        room = case["maxeval"] - state["done"] - len(R) * nnew
        K = min(len(order), case["width"], max(0, room // (3 * nnew)), case["max_regions"] - len(R))
        if K <= 0:
            break
        for k in order[:K]:
            e, axis = R[k][0], int(np.argmax(R[k][3]))
            left, right = e.copy(), e.copy()
            half = e[axis, :N // 2 + 1], e[axis, N // 2:]
            for child, q in zip((left, right), half):
                child[axis, 0::2] = q
                child[axis, 1::2] = 0.5 * (q[:-1] + q[1:])
            R[k] = adapt(left)
            R.append(adapt(right))
    last = [sample(r[0]) for r in R]
    I, V = sum(x[0] for x in last), sum(x[1] for x in last)
    boxes = np.stack([np.stack([r[0][:, 0], r[0][:, -1]], axis=1) for r in R])
    return dict(integral=I, error=np.sqrt(V), boxes=boxes, nregions=len(R), neval=state["done"], fail=1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        res = []
        for p in _many(case, seed):
            if kind == "batch":
                r = _vegas64(p, case["nbins"], 23, p["n"], 0, case["iters"] * p["n"])
            else:
                r = _vegas64(p, case["nbins"], 23, 10000, 50000, case["maxeval"], epsrel=p["epsrel"])
            res.append(r)
        nc = max(len(r["integral"]) for r in res)
        pad = lambda v: np.concatenate([v, np.zeros(nc - len(v))])  # noqa: E731
        return dict(integral=np.array([pad(r["integral"]) for r in res]),
                    error=np.array([pad(r["error"]) for r in res]), neval=None, fail=None)
    p, seed = _one(case, seed), int(seed) & 0x7fffffff
    bits = 52 if case.get("fp64") else 23
    if kind == "sample":
        S1, S2, H = _pass64(p, p["edges"], case["start"], case["n"], bits, case["gen"], seed)
        return dict(S1=S1, S2=S2, H=H.reshape(-1))
    if kind == "suave":
        if case["maxeval"] // case["nnew"] > 3000:  # (too many passes for a Python loop)
            return None
        r = _suave64(case, p)
        return dict(integral=r["integral"], error=r["error"], boxes=r["boxes"], nregions=None, neval=None, fail=None)
    r = _vegas64(p, case["nbins"], bits, case["nstart"], case["ninc"],
                 _maxeval(case["nstart"], case["ninc"], case["iters"]), case.get("gen", "sobol"), seed)
    keep = ["integral", "error"]
    if kind == "vegas" and case["fp64"]:
        keep.append("prob")
    if kind == "integral":
        keep += ["iterations", "variances", "grid"]
    return dict({k: r[k] for k in keep}, neval=None, fail=None)
