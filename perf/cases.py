"""What a user of this library has it do, as timed cases: the smallest calls
(a parameter scan of 1000-point estimates), ordinary runs, the workloads of
bench.py, odd sizes, both directions (estimate and gradient), the three
precision forms, stratified and plain sampling, batches, event generation,
run-time compiled integrands and the allocation-free pass.

A case is a dict of plain values:
  path       scan (new parameters, one estimate), vegas (refining iterations
             from the uniform grid), bases (both phases), grad (estimate and
             gradient through autograd), batch (many integrals at once),
             spring (events on a fixed grid), noalloc (one pass, caller's memory)
  integrand  the family, or "user" (CUDA source compiled at run time)
  ndim, nbins, ncall, nstrat, precision, ybits: as vegas_create takes them
  iters, iters2: iterations (of the second BASES phase)
  tuned      prepare() runs the autotuner, as bench.py does for this workload
  batch: instances, log2n_min, log2n_max;  spring: trials

Inputs (integrand parameters, Philox key) come from the seed alone.  The FP32
forms' outputs, accurate to FP32, are returned in FP32; the FP64 form's in
FP64.  `exact` restates the method in 64-bit torch and numpy.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1010_2107_gb300 import autograd as ag
from paper_1010_2107_gb300 import gvegas as gv
from paper_1010_2107_gb300 import workloads as wl

KINDS = {"gaussian": wl.GENZ_GAUSSIAN, "product_peak": wl.GENZ_PRODUCT_PEAK, "corner_peak": wl.GENZ_CORNER_PEAK,
         "oscillatory": wl.GENZ_OSCILLATORY, "double_gaussian": wl.DOUBLE_GAUSSIAN, "rambo": wl.RAMBO_BW,
         "continuous": wl.GENZ_CONTINUOUS, "discontinuous": wl.GENZ_DISCONTINUOUS, "wmunu": wl.W_MUNU}
NAMES = {v: k for k, v in KINDS.items()}
DIFFICULTY = {"oscillatory": 9.0, "product_peak": 7.25, "corner_peak": 1.85, "continuous": 20.0, "discontinuous": 4.0}

# A user's integrand: a Gaussian ridge times a slow wave, p = (centre, 1/width^2, amplitude, frequency).
USER_SOURCE = r"""
template <typename T>
__device__ T vegas_user_f(const T* x, int d, const T* p) {
  T q = T(0), s = T(0);
  for (int i = 0; i < d; ++i) {
    const T t = x[i] - p[0];
    q += t * t;
    s += x[i];
  }
  return exp(-q * p[1]) * (T(1) + p[2] * cos(p[3] * s));
}
"""


def case(path, integrand, ndim, ncall, *, nbins=50, nstrat=0, precision="fp32", ybits=0, **more):
    return dict(path=path, integrand=integrand, ndim=ndim, ncall=ncall, nbins=nbins, nstrat=nstrat,
                precision=precision, ybits=ybits, **more)


def listed():
    out = {
        # a fit's inner loop: new parameters, a small estimate, read back (latency)
        "scan_small": case("scan", "product_peak", 3, 1000),
        # the gauss4 workload of bench.py: the default precision (FP64), 5 x 1e5 points
        "gauss4": case("vegas", "gaussian", 4, 100_000, precision="fp64", iters=5),
        # an ordinary integral of odd dimension, bin count and point count
        "continuous6": case("vegas", "continuous", 6, 300_007, nbins=37, iters=4),
        # BASES in FP64 with a division count that is no power of two
        "bases3_fp64": case("bases", "gaussian", 3, 108_000, nstrat=6, precision="fp64", iters=3, iters2=3),
        # the dgauss8 workload of bench.py: BASES, 65 536 hypercubes, tuned as there
        "dgauss8": case("bases", "double_gaussian", 8, 1 << 22, nstrat=4, iters=5, iters2=5, tuned=True),
        # the wmunu workload of bench.py in the default launch shape
        "wmunu": case("bases", "wmunu", 5, 1 << 22, nbins=32, nstrat=8, iters=5, iters2=5),
        # the rambo5 workload's first iterations (20 dimensions, cuts; each refinement amplifies
        # the rounding of its heavy-tailed weights), tuned as in bench.py
        "rambo5": case("vegas", "rambo", 20, 1 << 24, iters=2, tuned=True),
        # the rambo4_adjoint workload: estimate and gradient in (M, Gamma, T)
        "rambo4_grad": case("grad", "rambo", 16, 1 << 24),
        # the genz256 workload: 256 integrals of 2..16 dimensions at once, tuned as in bench.py
        "genz256": case("batch", "mixed", 16, 0, instances=256, log2n_min=16.0, log2n_max=22.0, iters=3, tuned=True),
        # event generation on a fixed grid, events to pinned host memory
        "spring8": case("spring", "double_gaussian", 8, 1 << 22, nstrat=4, iters2=3, trials=1 << 22),
        # a user's own integrand, compiled at run time
        "user7": case("vegas", "user", 7, 1 << 20, iters=5),
        # one pass in the caller's own memory
        "noalloc10": case("noalloc", "corner_peak", 10, 262_147),
    }
    return [dict(c, name=n) for n, c in out.items()]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm (mostly odd ones)."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _strat(rng, d, nmax):
    """Divisions per axis and NCALL = g^d x points per hypercube."""
    g = rng.choice([g for g in (2, 3, 4, 5, 8, 16) if g ** d <= nmax // 8])
    return g, g ** d * _log(rng, 4, nmax // g ** d)


def draw(rng):
    """One more case: any path, any family it takes, sizes over the listed ones' range."""
    path = rng.choice(["scan", "vegas", "vegas", "bases", "bases", "grad", "batch", "batch", "spring", "noalloc"])
    nbins = rng.choice([32, 50, 50, 50, 64, rng.randint(10, 128)])
    prec = rng.choice(["fp32", "fp32", "fp32", "fp64", "fp32_acc64"])
    if path == "batch":
        hi = rng.uniform(12.0, 20.0)
        return case(path, "mixed", rng.randint(3, 16), 0, nbins=rng.choice([32, 50, 50]),
                    precision=rng.choice(["fp32", "fp32", "fp64"]), instances=_log(rng, 8, 200), log2n_min=10.0,
                    log2n_max=hi, iters=rng.randint(1, 3), tuned=False)
    if path == "grad":
        name = rng.choice(["rambo", "double_gaussian", "gaussian"])
        d = rng.choice([12, 16, 20]) if name == "rambo" else rng.randint(2, 16)
        prec = rng.choice(["fp32", "fp32", "fp64"])
        return case(path, name, d, _log(rng, 2000, 1 << (20 if prec == "fp64" else 23)), nbins=nbins, precision=prec)
    if path == "spring":
        d = rng.randint(3, 8)
        g, n = _strat(rng, d, 1 << 20)
        return case(path, "double_gaussian", d, n, nbins=50, nstrat=g, iters2=2, trials=_log(rng, 5000, 1 << 21))
    names = ["gaussian", "product_peak", "corner_peak", "oscillatory", "continuous", "discontinuous",
             "double_gaussian", "rambo", "wmunu"] + ([] if path == "noalloc" else ["user"])
    name = rng.choice(names)
    d = 5 if name == "wmunu" else 4 * rng.randint(2, 5) if name == "rambo" else rng.randint(1, 16)
    nmax = 1 << (18 if prec != "fp32" else 23)
    ybits = rng.choice([0, 0, 0, 53]) if prec != "fp64" else rng.choice([0, 0, 24])
    more = {}
    if path == "scan":
        n, g = _log(rng, 500, min(nmax, 1 << 20)), 0
    elif path == "bases":
        d = d if name in ("wmunu", "rambo") else rng.randint(1, 10)
        if name == "rambo":
            name, d = "double_gaussian", 8
        g, n = _strat(rng, d, nmax)
        g = g if g * nbins < 1024 else 2
        n = n if n % g ** d == 0 else g ** d * max(4, n // g ** d)
        more = dict(iters=rng.randint(1, 4), iters2=rng.randint(1, 4), tuned=False)
    else:
        n, g = _log(rng, nmax // 4 if name == "rambo" else 3000, nmax), 0  # cuts and a resonance need points
        if path == "vegas":
            more = dict(iters=1 if name == "rambo" else rng.randint(1, 3), tuned=rng.random() < 0.3)
    return case(path, name, d, n, nbins=nbins, nstrat=g, precision=prec, ybits=ybits, **more)


# ---------------------------------------------------------------- inputs
def _params(name, d, seed):
    """The integrand's parameter vector."""
    rng = np.random.Generator(np.random.PCG64([int(seed), d]))
    if name == "gaussian":
        return np.concatenate([rng.uniform(5.0, 10.0, d), rng.uniform(0.3, 0.7, d)])
    if name == "double_gaussian":
        return np.array([0.3 + 0.05 * rng.random(), 0.65 + 0.05 * rng.random(), 0.05])
    if name == "rambo":
        return wl.rambo_params(d // 4, cut=1 if d == 16 else 0, M=80.4 + 0.2 * rng.random())
    if name == "wmunu":
        return wl.w_munu_params(M=80.3 + 0.2 * rng.random())
    if name == "user":
        return np.array([rng.uniform(0.4, 0.6), 1.0 / 0.3 ** 2, 0.5, rng.uniform(1.0, 3.0)])
    a, u = 0.2 + rng.random(d), rng.uniform(0.2, 0.8, d)
    a *= DIFFICULTY[name] / a.sum()
    if name == "corner_peak":
        return a
    return np.concatenate([a, u[:1] if name == "oscillatory" else u[:2] if name == "discontinuous" else u])


def _instances(c, seed):
    """The batch's integrals: the draw of workloads.genz_batch with sizes and dimensions of the case."""
    return wl.genz_batch(c["instances"], seed=int(seed), dmax=c["ndim"], log2n_min=c["log2n_min"],
                         log2n_max=c["log2n_max"])


def _key(seed):
    return 1 + (int(seed) * 2654435761) % (1 << 40)


def _peaked_grid(p, d, N):
    """Edges [d][N+1] of equal share of 1/4 uniform + 3/4 two peaks: what a run's first phase leaves."""
    c1, c2, w = p
    x = np.linspace(0.0, 1.0, 20001)
    cdf = 0.25 * x + sum(0.375 * 0.5 * np.array([math.erf((v - c) / w) for v in x]) for c in (c1, c2))
    cdf = (cdf - cdf[0]) / (cdf[-1] - cdf[0])
    e = np.interp(np.arange(N + 1) / N, cdf, x)
    e[0], e[-1] = 0.0, 1.0
    return np.tile(e, (d, 1))


def prepare(c, seed):
    s = dict(case=c, out=np.float64 if c["precision"] == "fp64" else np.float32)
    kw = dict(nbins=c["nbins"], seed=_key(seed), precision=c["precision"], ybits=c["ybits"])
    if c["path"] == "batch":
        s["ctx"] = gv.vegas_batch_create(_instances(c, seed), **kw)
        if c.get("tuned"):
            gv.vegas_batch_autotune(s["ctx"])
        return s
    d, N = c["ndim"], c["nbins"]
    kw.update(ncall=c["ncall"], nstrat=c["nstrat"])
    p = s["params"] = _params(c["integrand"], d, seed)
    if c["path"] == "noalloc":
        edges = np.tile(np.arange(N + 1) / N, (d, 1))
        s["edges"] = torch.as_tensor(edges, device="cuda")
        s["buf"] = torch.zeros(2 * d * N + 5, dtype=torch.float64, device="cuda")
        s["kw"] = kw
        return s
    if c["integrand"] == "user":
        ctx = gv.vegas_create_user(USER_SOURCE, d, p, **kw)
    else:
        ctx = gv.vegas_create(KINDS[c["integrand"]], d, p, **kw)
    s["ctx"] = ctx
    if c.get("tuned"):
        gv.vegas_autotune(ctx)
    if c["path"] == "grad":
        slots = ag.theta_slots(KINDS[c["integrand"]], d)
        dt = torch.float64 if c["precision"] == "fp64" else torch.float32
        s["theta"] = torch.tensor(p[slots], dtype=dt, requires_grad=True)
    if c["path"] == "spring":
        gv.vegas_set_grid(ctx, _peaked_grid(p, d, N))
        gv.bases_integrate(ctx, 0, 0.0, c["iters2"], 0.0)
        s["x"] = torch.zeros((c["trials"], d), dtype=torch.float64, pin_memory=True).numpy()
        s["t"] = torch.zeros(c["trials"], dtype=torch.int64, pin_memory=True).numpy().view(np.uint64)
    return s


# ---------------------------------------------------------------- one pass
def _result(r, to):
    # (chi2_dof follows from the history, which is returned: where its estimates agree, their
    # differences are rounding)
    return dict(value=np.array([r["I"], r["sigma"]], to), iters=r["iters_done"], nonfinite=r["nonfinite"],
                samples=r["samples"])


def _grid(s):
    edges, bins = gv.vegas_get_grid(s["ctx"], bin_sums=True)
    return dict(edges=edges.astype(s["out"]), s1=bins[0].astype(s["out"]), s2=bins[1].astype(s["out"]))


def run(s):
    c, to = s["case"], s["out"]
    ctx = s.get("ctx")
    if c["path"] == "scan":
        gv.vegas_set_params(ctx, s["params"])
        return np.array(gv.vegas_eval(ctx, 0), to)
    if c["path"] in ("vegas", "bases"):
        gv.vegas_reset_grid(ctx)
        gv.vegas_set_iteration(ctx, 0)
        gv.vegas_reset_results(ctx)
        if c["path"] == "vegas":
            out = _result(gv.vegas_iterate(ctx, c["iters"]), to)
        else:
            r2, r1 = gv.bases_integrate(ctx, c["iters"], 0.0, c["iters2"], 0.0)
            out = dict(_result(r2, to), phase1=_result(r1, to))
        out["history"] = gv.vegas_get_history(ctx).astype(to)
        return dict(out, **_grid(s))
    if c["path"] == "grad":
        theta = s["theta"]
        theta.grad = None
        I = ag.vegas_estimate(theta, ctx, 0, s["params"], KINDS[c["integrand"]])
        I.backward()
        return dict(I=I.detach(), grad=theta.grad)
    if c["path"] == "batch":
        gv.vegas_batch_reset(ctx)
        rs = gv.vegas_batch_iterate(ctx, c["iters"])
        return dict(value=np.array([[r["I"], r["sigma"]] for r in rs], to),
                    samples=np.array([r["samples"] for r in rs]))
    if c["path"] == "spring":
        ev = gv.spring_generate(ctx, 0, c["trials"], out_x=s["x"], out_t=s["t"])
        return dict(x=s["x"], trial=s["t"].view(np.int64), n_events=ev["n_events"], overflow=ev["overflow"],
                    nonpos=ev["nonpos"])  # the caller's buffers: the events are their heads
    gv.vegas_eval_noalloc(KINDS[c["integrand"]], c["ndim"], s["params"], s["edges"].data_ptr(), 0,
                          s["buf"].data_ptr(), **s["kw"])
    b = s["buf"] if c["precision"] == "fp64" else s["buf"].float()
    dN = c["ndim"] * c["nbins"]
    return dict(s1=b[:dN], s2=b[dN:2 * dN], I=b[2 * dN:2 * dN + 1], var=b[2 * dN + 1:2 * dN + 2],
                sums=b[2 * dN + 2:2 * dN + 4], nonfinite=b[2 * dN + 4:])


# ---------------------------------------------------------------- work
# Operations per axis and per point of the integrands (a transcendental function counted as one).
_F_OPS = {"gaussian": (3, 2), "product_peak": (3, 2), "corner_peak": (2, 4), "oscillatory": (2, 3),
          "continuous": (3, 2), "discontinuous": (2, 4), "double_gaussian": (6, 6), "user": (4, 6),
          "rambo": (30, 60), "wmunu": (10, 40), "mixed": (2, 4)}


def _point_ops(name, d, yb, bins):
    axis, point = _F_OPS[name]
    # Philox: 10 rounds x 6 operations per four words; bin, fraction and map 11 per axis; sums 2 per axis and 14
    return 60 * math.ceil(d * (2 if yb == 53 else 1) / 4) + (11 + axis + (2 if bins else 0)) * d + point + 14


def work(c):
    yb = c["ybits"] or (53 if c["precision"] == "fp64" else 24)
    name, d, N = c["integrand"], c["ndim"], c["nbins"]
    esz = 8 if c["precision"] == "fp64" else 4
    if c["path"] == "batch":
        ins = _instances(c, 1)
        pts = sum(i["ncall"] * _point_ops("mixed", i["ndim"], yb, True) for i in ins)
        cells = sum(i["ndim"] * N for i in ins)
        return dict(flops=float(c["iters"] * pts), bytes=float(cells * 2 * esz + 24 * len(ins)))
    if c["path"] == "spring":
        ops = _point_ops(name, d, yb, False) + 70  # a third Philox block, the cube search, the decision
        return dict(flops=float(c["trials"] * ops), bytes=float(0.25 * c["trials"] * 8 * (d + 1) + 24 * c["nstrat"] ** d))
    frozen = c["ncall"] * _point_ops(name, d, yb, False)
    refining = c["ncall"] * _point_ops(name, d, yb, True)
    passes = {"scan": frozen, "grad": frozen + 20 * c["ncall"], "noalloc": refining,
              "vegas": c.get("iters", 0) * refining,
              "bases": c.get("iters", 0) * refining + c.get("iters2", 0) * frozen}[c["path"]]
    return dict(flops=float(passes), bytes=float(d * N * 2 * esz + 8 * d * (N + 1) + 64))


# ---------------------------------------------------------------- exact
_M32 = 0xFFFFFFFF


def _hilo(a, b):
    """The two halves of a 32 x 32 bit product (64-bit integers that wrap)."""
    p = a * b
    return (p >> 32) & _M32, p & _M32


def _philox(c0, c1, c2, c3, key):
    """Philox4x32-10 (Salmon et al., SC'11) on tensors of 64-bit integers."""
    k0, k1 = key & _M32, key >> 32
    for _ in range(10):
        h0, l0 = _hilo(0xD2511F53, c0)
        h1, l1 = _hilo(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


def _integrand(name, x, p):
    """f at the points x [n][d], in 64 bits; p: the parameter vector (a tensor)."""
    n, d = x.shape
    if name == "gaussian":
        return torch.exp(-((p[:d] * (x - p[d:])) ** 2).sum(1))
    if name == "product_peak":
        return 1.0 / (p[:d] ** -2 + (x - p[d:]) ** 2).prod(1)
    if name == "corner_peak":
        return (1.0 + x @ p) ** -(d + 1.0)
    if name == "oscillatory":
        return torch.cos(2 * math.pi * p[d] + x @ p[:d])
    if name == "continuous":
        return torch.exp(-((x - p[d:]).abs() @ p[:d]))
    if name == "discontinuous":
        inside = (x[:, :2] <= p[d:]).all(1)
        return torch.where(inside, torch.exp(x @ p[:d]), torch.zeros_like(x[:, 0]))
    if name == "double_gaussian":
        w = p[2]
        q = [((x - p[k]) ** 2).sum(1) / w ** 2 for k in (0, 1)]
        return 0.5 * (w * math.sqrt(math.pi)) ** -d * (torch.exp(-q[0]) + torch.exp(-q[1]))
    if name == "user":
        return torch.exp(-((x - p[0]) ** 2).sum(1) * p[1]) * (1 + p[2] * torch.cos(p[3] * x.sum(1)))
    return _wmunu(x, p) if name == "wmunu" else _rambo(x, p)


def _rambo(x, p):
    """Massless phase space (Kleiss, Stirling, Ellis 1986) x cuts x Breit-Wigner x prod 1/s_{i,i+1}, in GeV."""
    n, rs, M, G, ptmin, drmin, cut, T, wc = int(p[0]), p[1], p[2], p[3], p[4], p[5], int(p[6]), p[7], p[8]
    r = x.view(-1, n, 4)
    rho = r[..., 0] * r[..., 1]
    cth, phi, q0 = 2 * r[..., 2] - 1, 2 * math.pi * r[..., 3], -torch.log(rho.clamp(min=1e-300))
    sth = 2 * torch.sqrt(r[..., 2] * (1 - r[..., 2]))
    dirs = torch.stack([sth * torch.cos(phi), sth * torch.sin(phi), cth], -1)
    q = q0[..., None] * dirs
    Q0, Q = q0.sum(1), q.sum(1)
    m2 = torch.zeros_like(Q0)
    for i in range(n):
        for j in range(i + 1, n):
            m2 = m2 + q0[:, i] * q0[:, j] * ((dirs[:, i] - dirs[:, j]) ** 2).sum(-1)
    m = torch.sqrt(m2)
    b, gam = -Q / m[:, None], Q0 / m
    bq = (b[:, None] * q).sum(-1)
    k = (rs / m)[:, None, None] * (q + b[:, None] * (q0 + bq / (1 + gam)[:, None])[..., None])
    pt = torch.sqrt(k[..., 0] ** 2 + k[..., 1] ** 2)
    eta, az = torch.asinh(k[..., 2] / pt), torch.atan2(k[..., 1], k[..., 0])
    ok = (rho > 0).all(1).to(x.dtype)  # a zero uniform carries no weight
    if cut == 0:
        ok = ok * (pt > ptmin).all(1)
    elif cut == 1:
        ok = ok * torch.sigmoid((pt - T) / wc).prod(1)
    if cut != 2:
        for i in range(n):
            for j in range(i + 1, n):
                dphi = torch.remainder(az[:, i] - az[:, j] + math.pi, 2 * math.pi) - math.pi
                ok = ok * ((eta[:, i] - eta[:, j]) ** 2 + dphi ** 2 > drmin ** 2)
    s = rs * rs
    sij = [s * q0[:, i] * q0[:, j] * ((dirs[:, i] - dirs[:, j]) ** 2).sum(-1) / m2
           for i, j in ((i, (i + 1) % n) for i in range(n))]
    vol = (math.pi / 2) ** (n - 1) * s ** (n - 2) / (math.factorial(n - 1) * math.factorial(n - 2))
    f = ok * vol * M * G / ((sij[0] - M * M) ** 2 + (M * G) ** 2)
    for v in sij:
        f = f / v
    return f


def _wmunu(x, p):
    """u dbar -> W+ -> mu+ nu in pb with the lepton cuts; parton densities A x^a (1 - x)^b."""
    rs, M, G, gf, vud, ptmin, etamax, smin = (float(v) for v in p[:8])
    au, alu, bu, ad, ald, bd = (float(v) for v in p[9:15])
    S, M2 = rs * rs, M * M
    lo, hi = (math.atan((v - M2) / (M * G)) for v in (smin, S))
    shat = M2 + M * G * torch.tan(lo + (hi - lo) * x[:, 0])
    L = -torch.log(shat / S)
    y = (x[:, 1] - 0.5) * L
    x1, x2 = torch.exp(-L / 2 + y), torch.exp(-L / 2 - y)
    c = 2 * x[:, 2] - 1
    pt, eta = 0.5 * torch.sqrt(shat * (1 - c * c)), torch.atanh(c) + y
    ok = (pt > ptmin) & (eta.abs() < etamax) & (torch.floor(16 * x[:, 4]) == 10) & (x1 < 1) & (x2 < 1)
    g4 = (8 * M2 * gf / math.sqrt(2.0)) ** 2
    # flux x two-body phase space x averaged |M|^2 over the Breit-Wigner mapping's Jacobian
    lumi = au * x1 ** alu * (1 - x1) ** bu * ad * x2 ** ald * (1 - x2) ** bd
    k = (hi - lo) * g4 * vud * vud * 0.3893793721e9 / (48 * math.pi * S * M * G)
    return torch.where(ok, k * lumi * L * shat * (1 - c) ** 2, torch.zeros_like(L))


class _Exact:
    """The method in 64 bits: one integral's passes on a grid."""

    def __init__(self, name, d, n, nbins, nstrat, yb, key, p, instance=0):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.name, self.d, self.n, self.N, self.yb, self.key, self.inst = name, d, n, nbins, yb, key, instance
        self.g = max(nstrat, 1)
        self.G = self.g ** d
        self.nc = n // self.G
        self.p = torch.as_tensor(p, dtype=torch.float64, device=self.dev)
        chunk = max(1, (1 << 21) * 4 // max(4, d))
        self.chunk = chunk if self.G == 1 else self.nc * max(1, chunk // self.nc)

    def points(self, edges, it, s):
        """Bins, points and Jacobian of the samples s."""
        words, d, g, N, yb = [], self.d, self.g, self.N, self.yb
        for b in range((d * (1 if yb == 24 else 2) + 3) // 4):
            words += _philox(s, b, it, self.inst, self.key)
        cube = s // self.nc
        bins, xs, jac = [], [], torch.ones(len(s), dtype=torch.float64, device=self.dev)
        for a in range(d):
            m = words[a] >> 8 if yb == 24 else ((words[2 * a] >> 5) << 26) | (words[2 * a + 1] >> 6)
            t = (m if self.G == 1 else ((cube // g ** a % g) << yb) | m) * N
            k = t // (g << yb)
            fr = (t - k * (g << yb)).to(torch.float64) / float(g << yb)
            lo, w = edges[a][k], edges[a][k + 1] - edges[a][k]
            bins.append(k)
            xs.append(lo + fr * w)
            jac = jac * (N * w)
        return bins, torch.stack(xs, 1), jac

    def evaluate(self, edges, it, bins=True):
        """One pass: estimate, variance, sums of w and w^2, per-bin sums."""
        e = torch.as_tensor(edges, device=self.dev)
        sw = sw2 = si = sv = 0.0
        s12 = torch.zeros((2, self.d, self.N), dtype=torch.float64, device=self.dev)
        for s0 in range(0, self.n, self.chunk):
            s = torch.arange(s0, min(self.n, s0 + self.chunk), device=self.dev)
            kb, x, jac = self.points(e, it, s)
            w = _integrand(self.name, x, self.p) * jac
            w = torch.where(torch.isfinite(w), w, torch.zeros_like(w))
            sw, sw2 = sw + w.sum(), sw2 + (w * w).sum()
            if self.G > 1:
                v = w.view(-1, self.nc)
                m = v.mean(1)
                si = si + m.sum()
                sv = sv + (((v * v).mean(1) - m * m) / (self.nc - 1)).clamp(min=0).sum()
            for a in range(self.d if bins else 0):
                s12[0, a] += torch.bincount(kb[a], w, self.N)
                s12[1, a] += torch.bincount(kb[a], w * w, self.N)
        sw, sw2 = float(sw), float(sw2)
        if self.G > 1:
            I, var = float(si) / self.G, float(sv) / self.G ** 2
        else:
            I = sw / self.n
            var = max(0.0, (sw2 / self.n - I * I) / (self.n - 1))
        return I, var, sw, sw2, s12.cpu().numpy()

    def gradient(self, edges, it, slots):
        """The estimate and its derivative in the parameters `slots`."""
        e, I, g = torch.as_tensor(edges, device=self.dev), 0.0, 0.0
        theta = self.p[slots].clone().requires_grad_(True)
        p = self.p.clone()
        chunk = min(self.chunk, 1 << 19)
        for s0 in range(0, self.n, chunk):
            _, x, jac = self.points(e, it, torch.arange(s0, min(self.n, s0 + chunk), device=self.dev))
            q = list(p.unbind())
            for j, k in enumerate(slots):
                q[k] = theta[j]
            v = (_integrand(self.name, x, torch.stack(q)) * jac).sum()
            g = g + torch.autograd.grad(v, theta)[0]
            I = I + v.detach()
        return I / self.n, g / self.n


def _refine(edges, s2, alpha=1.5):
    """Lepage's grid optimisation (1978), one axis after another."""
    out = edges.copy()
    for a, d in enumerate(s2):
        N = len(d)
        if N == 2:
            sm = np.full(2, d.sum() / 2)
        else:
            sm = np.concatenate([[(d[0] + d[1]) / 2], (d[:-2] + d[1:-1] + d[2:]) / 3, [(d[-2] + d[-1]) / 2]])
        D = sm.sum()
        if not (D > 0 and np.isfinite(D)):
            continue
        y = sm / D
        with np.errstate(all="ignore"):
            r = np.where(y <= 0, 0.0, np.where(y >= 1, 1.0, ((1 - y) / -np.log(y)) ** alpha))
        C = np.concatenate([[0.0], np.cumsum(r)])
        tau = np.arange(1, N) * C[-1] / N
        k = np.minimum(np.searchsorted(C[1:], tau), N - 1)
        e = edges[a]
        out[a, 1:-1] = e[k] + (tau - C[k]) / r[k] * (e[k + 1] - e[k])
    return out


def _combine(hist):
    I, v = np.array([h[0] for h in hist]), np.array([h[1] for h in hist])
    W = (1 / v).sum()
    return dict(value=np.array([(I / v).sum() / W, W ** -0.5]), iters=None, nonfinite=None, samples=None)


def exact(c, seed):
    yb = c["ybits"] or (53 if c["precision"] == "fp64" else 24)
    N, key = c["nbins"], _key(seed)
    uniform = lambda d: np.tile(np.arange(N + 1) / N, (d, 1))  # noqa: E731
    if c["path"] == "spring":
        return None  # what is kept are decisions, the points themselves the sampling step's
    if c["path"] == "batch":
        out = []
        for i in _instances(c, seed):
            e, edges, hist = _Exact(NAMES[i["kind"]], i["ndim"], i["ncall"], N, 0, yb, key, i["params"],
                                    i["instance"]), uniform(i["ndim"]), []
            for it in range(c["iters"]):
                I, var, _, _, s12 = e.evaluate(edges, it, bins=it + 1 < c["iters"])
                hist.append((I, var))
                edges = _refine(edges, s12[1]) if it + 1 < c["iters"] else edges
            out.append(_combine(hist)["value"])
        return dict(value=np.array(out), samples=None)
    d = c["ndim"]
    p, edges = _params(c["integrand"], d, seed), uniform(d)
    e = _Exact(c["integrand"], d, c["ncall"], N, c["nstrat"], yb, key, p)
    if c["path"] == "scan":
        return np.array(e.evaluate(edges, 0, bins=False)[:2])
    if c["path"] == "grad":
        slots = ag.theta_slots(KINDS[c["integrand"]], d)
        # the gradient starts from the parameters the state's theta holds
        if c["precision"] != "fp64":
            e.p[slots] = e.p[slots].float().double()
        I, g = e.gradient(edges, 0, slots)
        return dict(I=I, grad=g)
    if c["path"] == "noalloc":
        I, var, sw, sw2, s12 = e.evaluate(edges, 0)
        return dict(s1=s12[0].ravel(), s2=s12[1].ravel(), I=np.array([I]), var=np.array([var]),
                    sums=np.array([sw, sw2]), nonfinite=None)
    hist, first = [], []
    for it in range(c["iters"]):
        I, var, _, _, s12 = e.evaluate(edges, it)
        hist.append((I, var))
        edges = _refine(edges, s12[1])
    out = _combine(hist)
    if c["path"] == "bases":
        first, hist = out, [e.evaluate(edges, c["iters"] + k, bins=False)[:2] for k in range(c["iters2"])]
        out = dict(_combine(hist), phase1=first)
    return dict(out, history=np.array(hist), edges=edges, s1=s12[0], s2=s12[1])
