"""Performance cases of the m-Cubes library: what its users have it do.

Three ways of use are covered, each through the public binding
(paper_2202_01753_gb300.mcubes):

* one integral at a time (`Context.integrate`, or the step-level calls that a
  program uses to look at the adapted grid), in double and in mixed
  precision, from a quick 1e4-call estimate, where launches count, to 1e9
  calls per iteration;
* many integrals in one call (`Context.integrate_batch`);
* a queue of requests in front of a continuous-batching server
  (`Server.run_stream`).

Sizes are those of the paper's test suite (f1..f6, f_A), of the benchmark's
named workloads and of their smaller versions in the tests.  `exact` restates
the method in 64 bits (torch and numpy only): counter-based words, exact bin
positions, the piecewise-linear map, cube moments, smoothed and compressed
rebinning, inverse-variance weights.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2202_01753_gb300 import mcubes

CONST, GAUSS, CORNER, OSC, PRODPEAK, C0, DISCONT, COSMO6, TABLE = range(9)

# integrand name -> (family id, lower and upper bound of the box on every axis)
INTEGRANDS = {
    "gauss": (GAUSS, 0.0, 1.0),        # product Gaussian, centre and widths drawn
    "corner": (CORNER, 0.0, 1.0),      # corner peak, slopes drawn
    "osc": (OSC, 0.0, 1.0),            # oscillatory, phase and frequencies drawn
    "f1": (OSC, 0.0, 1.0),             # cos(sum i x_i)
    "f2": (PRODPEAK, 0.0, 1.0),        # product peak
    "f3": (CORNER, 0.0, 1.0),          # (1 + sum i x_i)^-(d+1)
    "f4": (GAUSS, 0.0, 1.0),           # exp(-625 sum (x_i - 1/2)^2)
    "f5": (C0, 0.0, 1.0),              # exp(-10 sum |x_i - 1/2|)
    "f6": (DISCONT, 0.0, 1.0),         # exp(sum (i+4) x_i), cut at (3+i)/10
    "fA": (OSC, 0.0, 10.0),            # sin(sum x_i)
    "cosmo": (COSMO6, 0.05, 2.0),      # power laws x lognormal peak x ridge
    "table": (TABLE, 0.0, 1.0),        # interpolation tables
}


def _one(name, integrand, d, ncall, itmax, precision="fp64", kind="integrate", ita=-1, g=0, one_dim=0, rel_tol=0.0,
         knots=0):
    c = dict(kind=kind, integrand=integrand, d=d, ncall=ncall, itmax=itmax, ita=ita, g=g, one_dim=one_dim,
             precision=precision, rel_tol=rel_tol, knots=knots)
    return dict(c, name=name) if name else c


def _many(name, kind, n, precision, dmin, dmax, ncall_lo, ncall_hi, itmax, tol_lo, tol_hi):
    c = dict(kind=kind, n=n, precision=precision, dmin=dmin, dmax=dmax, ncall_lo=ncall_lo, ncall_hi=ncall_hi,
             itmax=itmax, tol_lo=tol_lo, tol_hi=tol_hi)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a quick look at a smooth integrand: the smallest call, launches and the rebinning count
        _one("gauss4_1e4_fp64", "gauss", 4, 10_000, 10),
        # the accuracy sweep's first level on the suite's f5
        _one("f5_d8_1e5_fp64", "f5", 8, 100_000, 10),
        # few cubes with many samples each (4 per axis), the grid and histogram read back between runs
        _one("gauss3_2e20_fp64", "gauss", 3, 2 ** 20, 10, kind="steps", g=4),
        # the suite's default size on its product peak
        _one("f2_d6_1e6_fp64", "f2", 6, 1_000_000, 10),
        # Table 1's f_A: adjusting iterations, then iterations on the frozen grid
        _one("fA_d6_1e7_fp64", "fA", 6, 10_000_000, 10, kind="steps", ita=5),
        # m-Cubes1D: one histogram serves every axis
        _one("f4_d6_1e7_onedim_fp64", "f4", 6, 10_000_000, 10, one_dim=1),
        # the cosmology-like integrand at its full size
        _one("cosmo6_1e8_fp64", "cosmo", 6, 100_000_000, 5),
        # an integrand that reads 285 MB of interpolation tables
        _one("table6_1e8_fp64", "table", 6, 100_000_000, 3, knots=4096),
        # mixed precision at 1e9 calls per iteration: the largest calls
        _one("corner8_1e9_mixed", "corner", 8, 1_000_000_000, 5, precision="mixed"),
        _one("osc10_1e9_mixed", "osc", 10, 1_000_000_000, 4, precision="mixed", kind="steps", ita=3),
        # uneven integrals to a tolerance, in one call
        _many("batch1024_mixed", "batch", 1024, "mixed", 2, 10, 10_000, 10_000_000, 10, 1e-4, 1e-4),
        # a burst of requests at the server
        _many("serve256_mixed", "serve", 256, "mixed", 3, 12, 100_000, 100_000, 20, 1e-5, 1e-3),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: an integral of the suite or of the drawn families (five times of eight), a table or cosmology
    integrand, a batch or a burst of requests."""
    what = rng.choice(["one", "one", "one", "one", "one", "sky", "batch", "serve"])
    if what == "one":
        name = rng.choice(["gauss", "corner", "osc", "f1", "f2", "f3", "f4", "f5", "f6", "fA"])
        precision = rng.choice(["fp64", "fp64", "mixed"])
        peaked = name in ("f2", "f4", "f6")  # their peaks want enough calls to be found, and few axes
        d = 6 if name == "fA" else rng.randint(2, 5 if peaked else 12)
        if precision == "mixed" and peaked:
            d = min(d, 3)  # narrower ones leave single precision's range
        itmax = rng.randint(2, 12)
        ita = rng.choice([-1, -1, max(1, itmax // 2)])
        one_dim = 1 if name in ("f2", "f4", "f5") and precision == "fp64" and rng.random() < 0.25 else 0
        top = 3e8 if precision == "mixed" else 5e7
        return _one("", name, d, _loguniform(rng, 2e5 if peaked else 1e4, top), itmax, precision=precision,
                    kind=rng.choice(["integrate", "steps"]), ita=ita, one_dim=one_dim)
    if what == "sky":
        if rng.random() < 0.6:
            return _one("", "cosmo", 6, _loguniform(rng, 1e5, 1e8), rng.randint(2, 5))
        return _one("", "table", 6, _loguniform(rng, 1e5, 5e7), rng.randint(2, 4), knots=rng.choice([257, 1024, 2048]))
    precision = rng.choice(["mixed", "mixed", "fp64"])
    if what == "batch":
        hi = _loguniform(rng, 1e5, 3e6)
        return _many("", "batch", _loguniform(rng, 8, 1024), precision, 2, rng.randint(3, 10), 10_000, hi,
                     rng.randint(4, 10), 1e-4, 1e-3)
    return _many("", "serve", _loguniform(rng, 2, 256), precision, 3, rng.randint(4, 12), 30_000, 100_000,
                 rng.randint(5, 20), 1e-5, 1e-3)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _params(name, d, rng):
    i = np.arange(1, d + 1, dtype=np.float64)
    if name == "gauss":
        return np.concatenate([[1.0], rng.uniform(0.3, 0.7, size=d), rng.uniform(0.1, 0.3, size=d)])
    if name == "corner":
        return rng.uniform(0.5, 2.0, size=d)
    if name == "osc":
        return np.concatenate([[rng.uniform(0.0, 1.0)], rng.uniform(0.5, 2.0, size=d)])
    if name == "f1":
        return np.concatenate([[0.0], i])
    if name == "f2":
        return np.concatenate([np.full(d, 50.0), np.full(d, 0.5)])
    if name == "f3":
        return i
    if name == "f4":
        return np.concatenate([[1.0], np.full(d, 0.5), np.full(d, math.sqrt(1.0 / 1250.0))])
    if name == "f5":
        return np.concatenate([np.full(d, 10.0), np.full(d, 0.5)])
    if name == "f6":
        return np.concatenate([i + 4.0, (3.0 + i) / 10.0])
    if name == "fA":
        return np.concatenate([[-0.25], np.ones(d)])
    if name == "cosmo":
        a = rng.uniform(0.2, 0.8, size=6)
        return np.concatenate([a, [math.log(0.5), 0.3, rng.uniform(0.8, 1.6), 0.01]])
    return np.array([1.0, 4.0, 0, 0, 1, 1, 2, -1, 2, 3, -1, 3, 4, 5])  # table: (table, axis, second axis) of each factor


def _tables(knots, rng):
    """Two bilinear and two linear tables: a Gaussian bump, a power law, a log-normal peak and a ridge."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    k2 = torch.linspace(0.0, 1.0, knots, dtype=torch.float64, device=dev)
    k1 = torch.linspace(0.0, 1.0, 256 * knots, dtype=torch.float64, device=dev)
    cx, cy = rng.uniform(0.3, 0.7, size=2)
    a, med, r = rng.uniform(0.2, 0.8), rng.uniform(0.3, 0.6), rng.uniform(0.8, 1.2)
    x, y = k2[:, None], k2[None, :]
    z = k1.clamp(min=1e-6)
    return [torch.exp(-((x - cx) ** 2 + (y - cy) ** 2) / (2 * 0.08 ** 2)) + 0.05,
            (k1 + 0.05) ** -a,
            torch.exp(-(torch.log(z / med) ** 2) / (2 * 0.3 ** 2)) / z + 1e-3,
            torch.exp(-((x + y - r) ** 2) / (2 * 0.03 ** 2)) + 1e-3]


def _input(case, seed):
    """Parameters, box and tables of a one-integral case."""
    rng = np.random.default_rng(seed)
    d = case["d"]
    fid, lo, hi = INTEGRANDS[case["integrand"]]
    p = _params(case["integrand"], d, rng)
    tabs = _tables(case["knots"], rng) if fid == TABLE else None
    return fid, p, np.full(d, lo), np.full(d, hi), tabs


def _requests(case, seed):
    rng = np.random.default_rng(seed)
    reqs = []
    for i in range(case["n"]):
        d = int(rng.integers(case["dmin"], case["dmax"] + 1))
        name = ["gauss", "corner", "osc"][int(rng.integers(0, 3))]
        ncall = int(round(math.exp(rng.uniform(math.log(case["ncall_lo"]), math.log(case["ncall_hi"])))))
        tol = math.exp(rng.uniform(math.log(case["tol_lo"]), math.log(case["tol_hi"])))
        reqs.append(dict(fid=INTEGRANDS[name][0], params=_params(name, d, rng), lo=np.zeros(d), hi=np.ones(d),
                         ncall=ncall, itmax=case["itmax"], rel_tol=tol, abs_tol=0.0, seed=seed * 65536 + i))
    return reqs


def prepare(case, seed):
    if case["kind"] in ("batch", "serve"):
        ctx = mcubes.Context(0, precision=case["precision"])
        s = dict(kind=case["kind"], ctx=ctx, reqs=_requests(case, seed))
        if case["kind"] == "serve":
            # a server with room for the whole burst; two iterations between looks at who is done
            probe = mcubes.Server(ctx, 1 << 20, case["itmax"])
            slot = probe.stats()["slot_bytes"]
            probe.close()
            s["server"] = mcubes.Server(ctx, slot * case["n"], case["itmax"])
            s["server"].set_step_iterations(2)
            s["arrivals"] = np.zeros(case["n"])
        return s
    fid, p, lo, hi, tabs = _input(case, seed)
    ctx = mcubes.Context(0, seed=seed, precision=case["precision"], ita=case["ita"], g_override=case["g"],
                         one_dim=case["one_dim"])
    if tabs is not None:
        ctx.set_tables([dict(ndim=t.dim(), values=t.cpu().numpy(), lo=(0.0,) * t.dim(), hi=(1.0,) * t.dim())
                        for t in tabs])
    return dict(kind=case["kind"], ctx=ctx, itmax=case["itmax"],
                args=(fid, p, lo, hi, case["ncall"], case["itmax"], case["rel_tol"]))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _columns(results):
    """The results of many integrals, a column for each field."""
    out = {k: np.array([r[k] for r in results], dtype=np.float64) for k in ("estimate", "sigma", "chi2_dof")}
    out.update({k: np.array([r[k] for r in results], dtype=np.int64)
                for k in ("iterations", "converged", "status", "samples_per_iter")})
    return out


def run(state):
    ctx = state["ctx"]
    if state["kind"] == "batch":
        return _columns(ctx.integrate_batch(state["reqs"]))
    if state["kind"] == "serve":
        return _columns(state["server"].run_stream(state["reqs"], state["arrivals"])[0])
    if state["kind"] == "steps":
        ctx.setup(*state["args"])
        ctx.iterate(state["itmax"])
        r = ctx.result()
    else:
        r = ctx.integrate(*state["args"])
    out = {k: r[k] for k in ("estimate", "sigma", "chi2_dof", "iterations", "converged", "samples_per_iter")}
    out["trace_I"], out["trace_V"] = ctx.trace(state["itmax"])
    if state["kind"] == "steps":
        out["grid"], out["hist"] = ctx.grid(), ctx.hist()
    return out


# ---------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------
NB = 500          # bins per axis (the library's default)
ALPHA = 1.5       # the rebinning's damping exponent


def _geometry(d, ncall, g_override=0):
    if g_override:
        g = g_override
    else:
        g = max(1, int((ncall // 2) ** (1.0 / d)))
        while (g + 1) ** d <= ncall // 2:
            g += 1
        while g > 1 and g ** d > ncall // 2:
            g -= 1
    m = g ** d
    return g, m, max(ncall // m, 2)


def _ops(d, adjust):
    """Integer and floating operations of one sample: per axis a quarter of a ten-round Philox block (15), the bin
    position (8), the map and its Jacobian (3), the integrand (4) and, adjusting, the histogram's addition (1); 20 for
    the integrand's end and the cube's moments."""
    return 20 + d * (30 + (1 if adjust else 0))


def work(case):
    """Operations of the samples that have to be drawn; bytes: parameters in, results, grid and histogram out, tables."""
    if case["kind"] in ("batch", "serve"):
        d = (case["dmin"] + case["dmax"]) / 2
        mean = case["ncall_lo"] if case["ncall_hi"] == case["ncall_lo"] else (
            (case["ncall_hi"] - case["ncall_lo"]) / math.log(case["ncall_hi"] / case["ncall_lo"]))
        its = 2  # a tolerance cannot be met earlier; how many more are needed depends on the integrand
        return {"bytes": case["n"] * (32 * d + 160), "flops": case["n"] * its * mean * _ops(d, True)}
    d = case["d"]
    _, m, p = _geometry(d, case["ncall"], case["g"])
    adj = case["itmax"] if case["ita"] < 0 else min(case["ita"], case["itmax"])
    b = 32 * d + 48 + 16 * case["itmax"] + (16 * d * NB if case["kind"] == "steps" else 0)
    if case["knots"]:
        b += 8 * (2 * case["knots"] ** 2 + 2 * 256 * case["knots"])
    return {"bytes": b, "flops": m * p * (adj * _ops(d, True) + (case["itmax"] - adj) * _ops(d, False))}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


class _F:
    """f(x), updated axis by axis."""

    def __init__(self, fid, p, d, tabs):
        self.fid, self.p, self.d, self.tabs = fid, p, d, tabs
        self.t, self.x = None, []

    def _add(self, v):
        self.t = v if self.t is None else self.t + v

    def add(self, j, x):
        p, d, fid = self.p, self.d, self.fid
        if fid == GAUSS:
            self._add((x - p[1 + j]) ** 2 / (2 * p[1 + d + j] ** 2))
        elif fid == CORNER:
            self._add(p[j] * x)
        elif fid == OSC:
            self._add(p[1 + j] * x)
        elif fid == PRODPEAK:
            v = 1.0 / (p[j] ** -2 + (x - p[d + j]) ** 2)
            self.t = v if self.t is None else self.t * v
        elif fid == C0:
            self._add(p[j] * (x - p[d + j]).abs())
        elif fid == DISCONT:
            self._add(torch.where(x < p[d + j], p[j] * x, -math.inf))
        elif fid == COSMO6:
            L = torch.log(x)
            v = p[j] * L
            if j in (2, 3):
                v = v + L + (L - p[6]) ** 2 / (2 * p[7] ** 2)
            self._add(v)
            if j < 2:
                self.x.append(x)
        else:
            self.x.append(x)

    def _interp(self, t, *xs):
        f, i = [], []
        for x, n in zip(xs, t.shape):
            u = x.clamp(0.0, 1.0) * (n - 1)
            k = u.floor().clamp(max=n - 2)
            f.append(u - k)
            i.append(k.long())
        if len(xs) == 1:
            return t[i[0]] * (1 - f[0]) + t[i[0] + 1] * f[0]
        a = t[i[0], i[1]] * (1 - f[0]) + t[i[0] + 1, i[1]] * f[0]
        b = t[i[0], i[1] + 1] * (1 - f[0]) + t[i[0] + 1, i[1] + 1] * f[0]
        return a * (1 - f[1]) + b * f[1]

    def end(self):
        p, fid, t = self.p, self.fid, self.t
        if fid == GAUSS:
            return p[0] * torch.exp(-t)
        if fid == CORNER:
            return (1 + t) ** -(self.d + 1.0)
        if fid == OSC:
            return torch.cos(2 * math.pi * p[0] + t)
        if fid == PRODPEAK:
            return t
        if fid == C0:
            return torch.exp(-t)
        if fid == DISCONT:
            return torch.exp(t)
        if fid == COSMO6:
            z = self.x[0] + self.x[1] - p[8]
            return torch.exp(-t - z * z / (2 * p[9] ** 2)) / (2 * math.pi * p[7] ** 2)
        x, T = self.x, self.tabs
        return p[0] * self._interp(T[0], x[0], x[1]) * self._interp(T[1], x[2]) * self._interp(T[2], x[3]) * \
            self._interp(T[3], x[4], x[5])


def _pass(case, seed, it, edges, inp, adjust, dev):
    """Sum of the cube means, of their variances, and the histograms of one sampling pass."""
    fid, prm, lo, hi, tabs = inp
    d = case["d"]
    g, m, p = _geometry(d, case["ncall"], case["g"])
    wide = np.diff(np.concatenate([np.zeros((d, 1), edges.dtype), edges], axis=1), axis=1)
    left = torch.from_numpy((edges - wide).astype(np.float64)).to(dev)
    width = torch.from_numpy(wide.astype(np.float64)).to(dev)
    nh = 1 if case["one_dim"] else d
    C = torch.zeros(d, NB, dtype=torch.float64, device=dev)
    s0 = torch.zeros((), dtype=torch.float64, device=dev)
    s1 = torch.zeros((), dtype=torch.float64, device=dev)
    step = max(1, (1 << 23) // p)
    for c0 in range(0, m, step):
        c1 = min(m, c0 + step)
        cube = torch.arange(c0, c1, device=dev).repeat_interleave(p)
        s = torch.arange(p, device=dev).repeat(c1 - c0)
        f, jac, rest, bins = _F(fid, prm, d, tabs), None, cube, []
        for j in range(d):
            if j % 4 == 0:
                w = _philox(s, cube, torch.full_like(s, it), torch.full_like(s, j // 4), seed)
            q = rest // g
            A = NB * (2 * w[j % 4] + 1)              # nb y = (nb c + A 2^-33) / g, exactly
            Q = NB * (rest - q * g) + (A >> 33)
            rest = q
            k = Q // g
            phi = ((Q - k * g).double() + (A & ((1 << 33) - 1)).double() * 2.0 ** -33) / g
            wk = width[j][k]
            f.add(j, float(lo[j]) + float(hi[j] - lo[j]) * (left[j][k] + wk * phi))
            v = wk * (NB * float(hi[j] - lo[j]))
            jac = v if jac is None else jac * v
            bins.append(k)
        F = f.end() * jac
        cubes = F.view(-1, p)
        mean = cubes.mean(dim=1)
        s0 += mean.sum()
        s1 += ((cubes - mean[:, None]) ** 2).sum() / (p * (p - 1.0))
        if adjust:
            for j in range(nh):
                C[j] += torch.bincount(bins[j], weights=F * F, minlength=NB)
    return float(s0), float(s1), C.cpu().numpy()


def _rebin(C, edges):
    """New right edges of one axis: bin sums smoothed over neighbours, normalised, compressed, equal shares."""
    sm = np.empty_like(C)
    sm[1:-1] = (C[:-2] + C[1:-1] + C[2:]) / 3
    sm[0], sm[-1] = (C[0] + C[1]) / 2, (C[-2] + C[-1]) / 2
    total = sm.sum()
    if not total > 0:
        return edges
    r = (sm / total).astype(np.longdouble)  # a share below the smallest double is none
    inner = (r > 0) & (r < 1)
    safe = np.where(inner, r, np.longdouble(0.5))
    w = np.where(inner, ((safe - 1) / np.log(safe)) ** np.longdouble(ALPHA), np.where(r >= 1, 1.0, 0.0))
    cum = np.cumsum(w)
    target = np.arange(1, NB).astype(np.longdouble) * cum[-1] / NB
    k = np.minimum(np.searchsorted(cum, target), NB - 1)
    before = np.where(k > 0, cum[k - 1], np.longdouble(0))
    left = np.where(k > 0, edges[k - 1], np.longdouble(0))
    return np.concatenate([left + (edges[k] - left) * (target - before) / w[k], np.ones(1, np.longdouble)])


def _weighted(I, V):
    w = 1.0 / V
    est = float((w * I).sum() / w.sum())
    chi2 = float((w * (I - est) ** 2).sum() / (len(I) - 1)) if len(I) > 1 else 0.0
    return est, float(1.0 / math.sqrt(w.sum())), chi2


def exact(case, seed):
    if case["kind"] in ("batch", "serve"):
        return None  # hundreds of integrals
    adj = case["itmax"] if case["ita"] < 0 else min(case["ita"], case["itmax"])
    if case["ncall"] * case["itmax"] * case["d"] > 4e9:
        return None  # longer than 20 seconds
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    inp = _input(case, seed)
    d = case["d"]
    g, m, p = _geometry(d, case["ncall"], case["g"])
    edges = np.tile(np.arange(1, NB + 1).astype(np.longdouble) / NB, (d, 1))
    I, V, C = [], [], np.zeros((d, NB))
    for it in range(case["itmax"]):
        a, b, h = _pass(case, seed, it, edges, inp, it < adj, dev)
        I.append(a / m)
        V.append(b / m / m)
        if it < adj:
            C = h
            edges = np.stack([_rebin(C[0 if case["one_dim"] else j], edges[j]) for j in range(d)])
    I, V = np.array(I), np.array(V)
    est, sigma, chi2 = _weighted(I, V)
    out = dict(estimate=est, sigma=sigma, chi2_dof=chi2, iterations=case["itmax"], converged=0, samples_per_iter=m * p,
               trace_I=I, trace_V=V)
    if case["kind"] == "steps":
        out["grid"], out["hist"] = edges.astype(np.float64), C
    return out
