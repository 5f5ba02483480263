"""The work that this library is used for, as cases that can be timed and compared.

A case is one pass of what a user's program does once it holds a context with its data:
an EM iteration, a whole fit, a log-likelihood, the posterior quantities of every pair,
the choice of starting values, an iteration on data that arrive anew, a batch of fits.
Sizes are those of the workloads of synth.py (two_comp_p2, flow_p4, wide_p16, learned_p6,
the ragged batch) at their full or a reduced number of observations, of the tests'
shapes, or odd ones between them.

Kinds of a pass (case["kind"]):
  em      set_params, estep, get_stats, mstep, get_params: one EM iteration whose
          statistics the program looks at
  fit     set_params, fit: `iters` EM iterations and the final log-likelihood
  score   set_params, loglik: the density-only pass
  pairs   set_params, estep, get_pairs: posteriors and conditional moments of every pair
  start   init from given partitions: the candidates of Algorithm 1
  stream  set_data (host FP32 rows), set_params, estep, mstep, get_params
  batch   set_params of every fit, fit_batch

The FP64 form's results are float64.  Those of the FP32 and mixed forms are taken on as
float32, the type that they were computed in.
"""
import math

import numpy as np
import torch

import paper_1606_02054_gb300 as cf
from paper_1606_02054_gb300 import synth

N_LATTICE, M_SHIFTS, KOROBOV = synth.DEFAULT_QMC_POINTS, synth.DEFAULT_QMC_SHIFTS, synth.DEFAULT_KOROBOV_A
LATTICE_SEED = synth.qmc_settings()["seed"]
PRECISIONS = {"fp64": cf.CFUST_PREC_FP64, "fp32": cf.CFUST_PREC_FP32, "mixed": cf.CFUST_PREC_MIXED}
NAMES = ("pi", "mu", "Sigma", "Delta", "nu")
NU_MIN, NU_MAX = 1.0, 200.0  # the library's default bracket


def _case(name, kind, p, q, g, n, precision, **more):
    return dict(name=name, kind=kind, p=p, q=q, g=g, n=n, precision=precision, moments=0, iters=1, **{}) | more


def listed():
    return [
        # a monitoring or model-selection script scores a few hundred new points under a
        # restricted skew t mixture (q = 1): the smallest call there is
        _case("score_p2_q1", "score", 2, 1, 2, 400, "fp64"),
        # a whole small fit with the default options: the two_comp_p2 workload
        _case("fit_two_comp_p2", "fit", 2, 2, 2, 1000, "fp64", iters=30),
        # starting values for a small problem, two partitions and the default alpha grid
        _case("start_p5_q2", "start", 5, 2, 3, 2503, "fp64", starts=2),
        # classification: the posteriors and moments of all pairs in FP64 (the single pass's
        # moments, which do not cancel in the tails of far components)
        _case("pairs_p3_q3", "pairs", 3, 3, 3, 1_201, "fp64", moments=1),
        # wide_p16 in the reference precision, a subsample as it is fitted before the full data
        _case("em_wide_p16_fp64", "em", 16, 2, 8, 20_000, "fp64"),
        # wide_p16 in the plain form: FP32 integrals, FP64 elsewhere
        _case("em_wide_p16_fp32", "em", 16, 2, 8, 200_000, "fp32"),
        # wide_p16 at full size in its chosen form
        _case("em_wide_p16_mixed", "em", 16, 2, 8, 2_000_000, "mixed"),
        # flow_p4 at full size in its chosen form (single-pass moments)
        _case("em_flow_p4_single", "em", 4, 4, 4, 200_000, "fp32", moments=1),
        # flow_p4 with the default moments (recursion through T_3 and T_2)
        _case("em_flow_p4_recursion", "em", 4, 4, 4, 20_000, "fp32"),
        # learned_p6 with single-pass moments in the mixed form
        _case("em_learned_p6_single", "em", 6, 6, 6, 50_000, "mixed", moments=1),
        # an odd size between the workloads, its rows new in every pass
        _case("stream_p7_q2", "stream", 7, 2, 3, 30_011, "mixed"),
        # ragged fits of the batched form, p = q from 2 to 8
        _case("batch_ragged", "batch", 8, 8, 6, 8_000, "fp32", moments=1, iters=3, fits=8, shapes=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(case):
    """Arithmetic of a pass, an FP64 operation counted as the 64 FP32 ones it costs here."""
    return work(case)["flops"] * (64 if case["precision"] == "fp64" else 1)


def draw(rng):
    kind = rng.choice(["score", "fit", "start", "pairs", "em", "em", "em", "em", "stream", "batch"])
    g = rng.randint(1, 8)
    more = {}
    if kind in ("score", "fit", "start"):
        q = rng.randint(1, 2)
        p = rng.randint(max(2, q), 6)
        precision, g = "fp64", rng.randint(2, 4)
        n = _log_int(rng, 400, 6000)
        if kind == "fit":
            more["iters"] = rng.randint(10, 30)
        if kind == "start":
            more["starts"] = rng.randint(1, 2)
    elif kind == "pairs":
        q = rng.randint(3, 4)
        p, precision, g, n = rng.randint(q, 6), "fp64", rng.randint(2, 4), _log_int(rng, 200, 1200)
        more["moments"] = 1
    elif kind == "batch":
        p = q = rng.randint(4, 8)
        precision, g, n = "fp32", rng.randint(3, 6), _log_int(rng, 2000, 8000)
        more.update(moments=1, iters=rng.randint(2, 3), fits=rng.randint(3, 8), shapes=rng.randint(2, 999))
    else:
        form = rng.choice(["fp64", "fp32", "mixed", "mixed", "single", "single", "recursion", "default"])
        if kind == "stream":
            form = "mixed"
        if form == "default":  # the library's default options at q = 3
            q, precision, n = 3, "fp64", _log_int(rng, 300, 1000)
            p, g = rng.randint(3, 5), min(g, 4)
        elif form in ("single", "recursion"):
            q = rng.randint(3, 6 if form == "single" else 4)
            p, precision = rng.randint(q, 8), rng.choice(["fp32", "mixed"])
            more["moments"] = 1 if form == "single" else 0
            n = _log_int(rng, 2000, 200_000)
        else:
            q = rng.choice([1, 2, 2, 2])
            p, precision = rng.randint(2, 20), form
            n = _log_int(rng, 2000, 20_000 if form == "fp64" else 500_000)
    case = _case("", kind, p, q, g, n, precision, **more)
    del case["name"]
    cap = max(_cost(c) for c in listed())
    while _cost(case) > 0.8 * cap or case["n"] * case["p"] * case["g"] > 60_000_000:
        case["n"] = max(100, int(case["n"] * 0.6))
    return case


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _shapes(case):
    """(p, q, g, n) of the fits of a pass: one, or the batch's."""
    if case["kind"] != "batch":
        return [(case["p"], case["q"], case["g"], case["n"])]
    r = np.random.default_rng([1606, case["shapes"]])
    out = []
    for i in range(case["fits"]):  # the first one is the largest named by the case
        p = case["p"] if i == 0 else int(r.integers(2, case["p"] + 1))
        g = case["g"] if i == 0 else int(r.integers(2, case["g"] + 1))
        n = int(round(math.exp(r.uniform(math.log(1000), math.log(case["n"])))))
        out.append((p, p, g, n))
    return out


def _inputs(case, seed):
    """Per fit: observations drawn from the mixture (eq 6), and parameters as a fit holds
    them some iterations in: near the drawn ones, but not at them."""
    out = []
    for i, (p, q, g, n) in enumerate(_shapes(case)):
        rng = np.random.default_rng([int(seed), i])
        truth = synth.draw_params(rng, p, q, g, mu_range=3.0 if p >= 12 else 5.0, wishart_df=max(8, 2 * p))
        truth["pi"] = 0.7 * truth["pi"] + 0.3 / g
        y, z = synth.sample(rng, n, truth, dtype=np.float64 if case["precision"] == "fp64" else np.float32)
        now = dict(pi=0.8 * truth["pi"] + 0.2 / g,
                   mu=truth["mu"] + 0.15 * rng.standard_normal((g, p)),
                   Sigma=1.15 * truth["Sigma"],
                   Delta=0.9 * truth["Delta"] + 0.1 * rng.standard_normal((g, p, q)),
                   nu=np.minimum(1.3 * truth["nu"], 60.0))
        fit = dict(p=p, q=q, g=g, n=n, y=y, params=now)
        if case["kind"] == "start":  # partitions: the drawn components with some labels changed
            flip = rng.random((case["starts"], n)) < 0.15
            fit["labels"] = np.where(flip, rng.integers(0, g, size=(case["starts"], n)), z[None, :]).astype(np.int32)
        out.append(fit)
    return out


def prepare(case, seed):
    fits = _inputs(case, seed)
    opts = cf.cfust_default_opts(precision=PRECISIONS[case["precision"]], moments=case["moments"],
                                 qmc_points=N_LATTICE, qmc_shifts=M_SHIFTS, qmc_korobov_a=KOROBOV, seed=LATTICE_SEED)
    ctxs = []
    for f in fits:
        ctx = cf.cfust_create(f["p"], f["q"], f["g"], f["n"], opts)
        if case["kind"] != "stream":
            cf.cfust_set_data(ctx, f["y"])
        ctxs.append(ctx)
    state = dict(case=dict(case), ctxs=ctxs, params=[f["params"] for f in fits])
    if case["kind"] == "stream":
        state["rows"] = torch.from_numpy(fits[0]["y"]).pin_memory()
    if case["kind"] == "start":
        state["labels"] = fits[0]["labels"]
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _typed(case, out):
    """float64 results as they are, those of the FP32 forms as float32."""
    if case["precision"] == "fp64":
        return out
    return {k: v if v.dtype.kind in "iu" else v.astype(np.float32) for k, v in out.items()}


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    ctxs, params = state["ctxs"], state["params"]
    ctx = ctxs[0]
    if kind == "batch":
        for c, p in zip(ctxs, params):
            cf.cfust_set_params(c, p)
        iters, hist, status = cf.cfust_fit_batch(ctxs, case["iters"])
        out = dict(iters=iters, status=status, hist=hist)
        for k in NAMES:
            out[k] = []
        for c in ctxs:
            got = cf.cfust_get_params(c)
            for k in NAMES:
                out[k].append(got[k].ravel())
        for k in NAMES:
            out[k] = np.concatenate(out[k])
        return _typed(case, out)
    if kind == "start":
        table, best = cf.cfust_init(ctx, nstarts=case["starts"], labels=state["labels"])
        return _typed(case, dict(cf.cfust_get_params(ctx), table=table, best=np.array([best])))
    if kind == "stream":
        cf.cfust_set_data(ctx, state["rows"])
    cf.cfust_set_params(ctx, params[0])
    if kind == "score":
        return _typed(case, dict(loglik=np.array([cf.cfust_loglik(ctx)])))
    if kind == "fit":
        iters, hist = cf.cfust_fit(ctx, case["iters"])
        return _typed(case, dict(cf.cfust_get_params(ctx), iters=np.array([iters]), hist=hist))
    loglik = cf.cfust_estep(ctx)
    if kind == "pairs":
        return _typed(case, dict(cf.cfust_get_pairs(ctx), loglik=np.array([loglik])))
    out = dict(loglik=np.array([loglik]))
    if kind == "em":
        out["stats"] = cf.cfust_get_stats(ctx)
    cf.cfust_mstep(ctx)
    out.update(cf.cfust_get_params(ctx))
    return _typed(case, out)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# floating-point operations of a normal CDF, its inverse, a node of the bivariate t CDF's
# quadrature (32 nodes taken for one) and a univariate t CDF
PHI, PHI_INV, T2_NODE, T2_NODES, T1 = 24, 26, 60, 32, 60


def _integral_flops(k):
    if k <= 0:
        return 0
    if k == 1:
        return T1
    if k == 2:
        return T2_NODES * T2_NODE
    return N_LATTICE * M_SHIFTS * (k * PHI + (k - 1) * PHI_INV + k * (k - 1) + 4 * k)


def _pair_flops(p, q, moments, density_only):
    white = p * (p + 1) + 2 * p * q + 3 * p + 20
    if density_only:
        return white + _integral_flops(q)
    stats = 2 * (3 + p + q + p * q + q * (q + 1) // 2 + p * (p + 1) // 2)
    if moments == 1 and q >= 3:
        point = q * (PHI + PHI_INV) + q * (q - 1) + 4 * q + 2 * (2 + q + q * (q + 1) // 2)
        return white + stats + N_LATTICE * M_SHIFTS * point
    integrals = 2 * _integral_flops(q) + q * _integral_flops(q - 1) + q * (q - 1) * _integral_flops(q - 2)
    return white + stats + integrals


def work(case):
    kind = case["kind"]
    size = 8 if case["precision"] == "fp64" else 4
    by = fl = 0.0
    for p, q, g, n in _shapes(case):
        par = 8.0 * g * (2 + p + p * q + p * p)
        stats = 8.0 * g * (3 + p + q + p * q + q * q + p * p)
        steps = case["iters"] if kind in ("fit", "batch") else 1
        one = g * n * float(_pair_flops(p, q, case["moments"], kind in ("score", "start")))
        if kind == "start":
            steps = 9 * case["starts"]
        rows = float(n) * p * size
        by += steps * (rows + 2 * par) + (stats if kind == "em" else 0)
        fl += steps * one
        if kind in ("fit", "batch"):  # the final log-likelihood
            by += rows
            fl += g * n * float(_pair_flops(p, q, case["moments"], True))
        if kind == "pairs":
            by += 8.0 * g * n * (5 + q + q * q)
        if kind == "stream":
            by += rows
        if kind == "start":
            by += 4.0 * case["starts"] * n
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _t(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device=_device())


def _legendre(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return _t(0.5 * (x + 1.0)), _t(0.5 * w)


def _t_const(nu):
    return math.exp(math.lgamma(0.5 * (nu + 1)) - math.lgamma(0.5 * nu)) / math.sqrt(math.pi)


def _t1(x, nu, nodes=40):
    """Student t CDF at dof nu: the angle phi = pi/2 + atan(x / sqrt nu), whose density is
    proportional to sin^(nu-1) phi, integrated from the nearer end."""
    u, w = _legendre(nodes)
    top = torch.atan2(torch.full_like(x, math.sqrt(nu)), x.abs())
    tail = torch.zeros_like(x)
    for i in range(nodes):
        tail += w[i] * torch.exp((nu - 1.0) * torch.log(torch.sin(top * u[i])))
    tail *= top * _t_const(nu)
    return torch.where(x > 0, 1.0 - tail, tail)


def _t2(h, k, rho, nu, nodes=48):
    """Bivariate t CDF: the first variable in the angle of _t1, the second one's conditional
    CDF inside, the interval cut where that one's argument changes sign."""
    sn = math.sqrt(nu)
    s = math.sqrt((nu + 1.0) / ((1.0 - rho * rho) * nu))
    top = 0.5 * math.pi + torch.atan(h / sn)
    cut = torch.atan2(torch.full_like(k, abs(rho) * sn), -math.copysign(1.0, rho) * k)
    cut = torch.minimum(cut, top)
    u, w = _legendre(nodes)
    out = torch.zeros_like(h)
    for lo, hi in ((cut, torch.zeros_like(cut)), (cut, top)):  # nodes denser towards the cut
        for i in range(nodes):
            phi = lo + (hi - lo) * u[i] ** 2
            arg = s * (k * torch.sin(phi) + rho * sn * torch.cos(phi))
            f = torch.exp((nu - 1.0) * torch.log(torch.sin(phi))) * _t1(arg, nu + 1.0)
            out += w[i] * 2.0 * u[i] * (hi - lo).abs() * torch.where(hi == lo, torch.zeros_like(f), f)
    return out * _t_const(nu)


def _u01(key):
    m = (1 << 64) - 1
    z = (key + 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return float((z ^ (z >> 31)) >> 11) / 9007199254740992.0


def _coordinates(d):
    """Coordinate d of every lattice point under every shift, after the baker's transform,
    and its complement."""
    z = pow(KOROBOV, d, N_LATTICE)
    i = (np.arange(N_LATTICE, dtype=np.int64) * z % N_LATTICE) / N_LATTICE
    x = np.concatenate([i + _u01(LATTICE_SEED ^ ((m + 1) << 32) ^ (d + 1)) for m in range(M_SHIFTS)])
    x = np.where(x >= 1.0, x - 1.0, x)
    far = np.abs(2.0 * x - 1.0)
    return _t(1.0 - far), _t(far)


def _chi(nu):
    """sqrt(chi-square quantile / nu) at coordinate 0 of the lattice."""
    w, wc = _coordinates(0)
    a = torch.full_like(w, 0.5 * nu)
    lo, hi = torch.zeros_like(w), torch.full_like(w, 40.0 * nu + 400.0)
    x = torch.full_like(w, nu)
    for _ in range(80):  # safeguarded Newton on the nearer tail
        h = 0.5 * x
        up = w > 0.5
        miss = torch.where(up, wc - torch.special.gammaincc(a, h), torch.special.gammainc(a, h) - w)
        hi = torch.where(miss > 0, x, hi)
        lo = torch.where(miss > 0, lo, x)
        dens = 0.5 * torch.exp((a - 1.0) * torch.log(h) - h - torch.lgamma(a))
        new = x - miss / dens
        x = torch.where((new > lo) & (new < hi), new, 0.5 * (lo + hi))
    return torch.sqrt(x / nu)


def _lattice(b, L, nu, moments, coords):
    """T_k over the lattice: mean f, and with moments also mean f s^2 and the f s^2-weighted
    means of X and X X^T at nu + 2 dof (standardised)."""
    K = b.shape[1]
    s = _chi(nu)
    step = max(1, (1 << 27) // (s.numel() * (K + 4)))
    rk = math.sqrt((nu + 2.0) / nu)
    low, high = 1e-300, 1.0 - 2.0 ** -53
    res = []
    for at in range(0, b.shape[0], step):
        bb = b[at:at + step]
        f, ys = None, []
        for r in range(K):
            a = bb[:, r:r + 1] * s
            for l in range(r):
                a -= L[r, l] * ys[l]
            e = torch.special.ndtr(a / L[r, r])
            f = e if f is None else f * e
            if r < K - 1 or moments:
                ys.append(torch.special.ndtri((coords[r] * e).clamp(low, high)))
        one = [f.mean(1)]
        if moments:
            one.append((f * s * s).mean(1))
            y = torch.stack(ys, 1)
            m1 = torch.einsum("nrs,ns->nr", y, f * s) * rk
            m2 = torch.bmm(y * f[:, None, :], y.transpose(1, 2)) * rk * rk
            tot = (f * s * s).sum(1)
            one.append((m1 / tot[:, None]) @ L.T)
            one.append(L @ (m2 / tot[:, None, None]) @ L.T)
        res.append(one)
    return [torch.cat(v) for v in zip(*res)]


def _corr(S):
    d = torch.sqrt(torch.diagonal(S))
    return d, torch.linalg.cholesky(S / d[:, None] / d[None, :])


def _tk(b, S, nu, coords):
    """T_k(b; 0, S, nu) for rows b that are scaled by their own factors already."""
    k = b.shape[1]
    if k == 0:
        return torch.ones(b.shape[0], dtype=b.dtype, device=b.device)
    d, L = _corr(S)
    b = b / d
    if k == 1:
        return _t1(b[:, 0], nu)
    if k == 2:
        return _t2(b[:, 0], b[:, 1], float(L[1, 0]), nu)
    return _lattice(b, L, nu, False, coords)[0]


def _logt1(x, v, nu):
    c = math.lgamma(0.5 * (nu + 1)) - math.lgamma(0.5 * nu) - 0.5 * math.log(nu * math.pi)
    return c - 0.5 * torch.log(v) - 0.5 * (nu + 1.0) * torch.log1p(x * x / (nu * v))


def _component(y, P, h, moments, density_only, coords):
    """log f, u, E log w, E2, E3 of every observation under component h (eqs 4, 13, 15-17)."""
    mu, Sg, Dl, nu = P["mu"][h], P["Sigma"][h], P["Delta"][h], float(P["nu"][h])
    p, q = Dl.shape
    r = y - mu
    Om = Sg + Dl @ Dl.T
    C = torch.linalg.cholesky(Om)
    z = torch.linalg.solve_triangular(C, r.T, upper=False).T
    d = (z * z).sum(1)
    A = torch.linalg.solve_triangular(C, Dl, upper=False)
    c = z @ A
    Lam = torch.eye(q, dtype=y.dtype, device=y.device) - A.T @ A
    logtp = (math.lgamma(0.5 * (nu + p)) - math.lgamma(0.5 * nu) - 0.5 * p * math.log(nu * math.pi)
             - torch.log(torch.diagonal(C)).sum() - 0.5 * (nu + p) * torch.log1p(d / nu))
    nu1 = nu + p
    b0 = c * torch.sqrt(nu1 / (nu + d))[:, None]
    single = moments == 1 and q >= 3
    if single and not density_only:
        dq, L = _corr(Lam)
        al_s, al, m1, m2 = _lattice(b0 / dq, L, nu1, True, coords)
    else:
        al_s = _tk(b0, Lam, nu1, coords)
    logf = q * math.log(2.0) + logtp + torch.log(al_s)
    if density_only:
        return (logf,)
    if not single:
        al = _tk(c * torch.sqrt((nu1 + 2.0) / (nu + d))[:, None], Lam, nu1 + 2.0, coords)
    u = nu1 / (nu + d) * al / al_s
    psi = float(torch.special.digamma(torch.tensor(0.5 * nu1, dtype=torch.float64)))
    elogu = u - torch.log(0.5 * (nu + d)) - nu1 / (nu + d) + psi
    if single:
        sig = torch.sqrt((nu + d) / (nu1 + 2.0))[:, None] * dq
        m1 = sig * m1
        m2 = sig[:, :, None] * sig[:, None, :] * m2
        eu = u[:, None] * (c - m1)
        cc = c[:, :, None] * c[:, None, :] - c[:, :, None] * m1[:, None, :] - m1[:, :, None] * c[:, None, :]
        return logf, u, elogu, eu, u[:, None, None] * (cc + m2)
    k0 = (nu + d) / nu1
    xi = torch.zeros_like(c)
    H = torch.zeros(c.shape[0], q, q, dtype=y.dtype, device=y.device)
    for a in range(q):
        oth = [i for i in range(q) if i != a]
        Saa = k0 * Lam[a, a]
        mv = Lam[oth, a] / Lam[a, a]
        sch = Lam[oth][:, oth] - torch.outer(Lam[oth, a], Lam[a, oth]) / Lam[a, a]
        cp = c[:, oth] - mv * c[:, a:a + 1]
        sc = (nu1 + c[:, a] ** 2 / Saa) / (nu1 + 1.0) * k0
        t1q = _tk(cp / torch.sqrt(sc)[:, None], sch, nu1 + 1.0, coords)
        xi[:, a] = torch.exp(_logt1(c[:, a], Saa, nu1)) * t1q
        H[:, a, a] = c[:, a] * xi[:, a]
        nu2 = nu1 + 1.0
        kp = nu2 / (nu2 - 2.0) * sc
        xp = torch.zeros_like(cp)
        for i in range(q - 1):
            ot2 = [k for k in range(q - 1) if k != i]
            V = kp * sch[i, i]
            m2v = sch[ot2, i] / sch[i, i]
            s2 = sch[ot2][:, ot2] - torch.outer(sch[ot2, i], sch[i, ot2]) / sch[i, i]
            ka = (nu2 - 2.0 + cp[:, i] ** 2 / V) / (nu2 - 1.0)
            b2 = (cp[:, ot2] - m2v * cp[:, i:i + 1]) / torch.sqrt(ka * kp)[:, None]
            xp[:, i] = torch.exp(_logt1(cp[:, i], V, nu2 - 2.0)) * _tk(b2, s2, nu1, coords)
        for j, b in enumerate(oth):
            v = xi[:, a] * (mv[j] * c[:, a] - kp * (xp @ sch[j]) / t1q)
            H[:, a, b] = torch.where(xi[:, a] == 0, torch.zeros_like(v), v)
    Lx = xi @ Lam
    eu = u[:, None] * c + Lx / al_s[:, None]
    LH = torch.einsum("ak,nkb->nab", Lam, H)
    cl = c[:, :, None] * Lx[:, None, :]
    euu = (u[:, None, None] * c[:, :, None] * c[:, None, :] + Lam
           + (cl + cl.transpose(1, 2) - 0.5 * (LH + LH.transpose(1, 2))) / al_s[:, None, None])
    return logf, u, elogu, eu, euu


def _estep(y, P, moments, density_only=False):
    q = P["Delta"].shape[2]
    coords = [_coordinates(d)[0] for d in range(1, q + 1)] if q >= 3 else None
    comp = [_component(y, P, h, moments, density_only, coords) for h in range(len(P["nu"]))]
    logf = torch.stack([c[0] for c in comp])
    lp = logf + torch.log(P["pi"])[:, None]
    lj = torch.logsumexp(lp, 0)
    pairs = dict(logf=logf, tau=torch.exp(lp - lj))
    if not density_only:
        null = torch.isinf(logf)  # T_q is 0 in 64 bits: u = 1, the others 0
        for k, v in zip(("u", "elogu", "eu", "euu"), zip(*[c[1:] for c in comp])):
            v = torch.stack(v)
            at = null.view(null.shape + (1,) * (v.dim() - 2))
            pairs[k] = torch.where(at, torch.full_like(v, 1.0 if k == "u" else 0.0), v)
    return lj.sum(), pairs


def _stats(y, P, E):
    out = []
    for h in range(len(P["nu"])):
        t, u, r = E["tau"][h], E["u"][h], y - P["mu"][h]
        tu = t * u
        out.append(torch.cat([t.sum()[None], tu.sum()[None], (t * (E["elogu"][h] - u)).sum()[None], tu @ r,
                              t @ E["eu"][h], ((t[:, None] * r).T @ E["eu"][h]).ravel(),
                              torch.einsum("n,nab->ab", t, E["euu"][h]).ravel(), ((tu[:, None] * r).T @ r).ravel()]))
    return torch.stack(out)


def _mstep(S, P, n):
    """Eqs 18-22 from the statistics."""
    new = {k: v.clone() for k, v in P.items()}
    p, q = P["Delta"].shape[1:]
    for h in range(S.shape[0]):
        s = S[h]
        N, U, Sn = s[0], s[1], s[2]
        at = 3
        part = []
        for size in (p, q, p * q, q * q, p * p):
            part.append(s[at:at + size])
            at += size
        Sr, Se, Sre, See, Srr = part[0], part[1], part[2].view(p, q), part[3].view(q, q), part[4].view(p, p)
        De = (Sr - P["Delta"][h] @ Se) / U
        A = Sre - torch.outer(De, Se)
        D = torch.linalg.solve(0.5 * (See + See.T), A.T).T
        Sg = (Srr - torch.outer(Sr, De) - torch.outer(De, Sr) + U * torch.outer(De, De) - D @ A.T - A @ D.T
              + D @ (0.5 * (See + See.T)) @ D.T) / N
        new["pi"][h], new["mu"][h], new["Delta"][h], new["Sigma"][h] = N / n, P["mu"][h] + De, D, 0.5 * (Sg + Sg.T)
        lo, hi = NU_MIN, NU_MAX
        bar = float(Sn / N)
        for _ in range(100):
            mid = 0.5 * (lo + hi)
            f = math.log(0.5 * mid) - float(torch.special.digamma(torch.tensor(0.5 * mid, dtype=torch.float64))) + 1.0 + bar
            lo, hi = (mid, hi) if f > 0 else (lo, mid)
        new["nu"][h] = 0.5 * (lo + hi)
    return new


def _starts(y, labels, g, q):
    """Eq 23 for every partition and alpha = 0.1 ... 0.9: the parameters."""
    for lab in labels:
        for a in range(1, 10):
            al = 0.1 * a
            P = dict(pi=[], mu=[], Sigma=[], Delta=[], nu=[])
            for h in range(g):
                yc = y[lab == h]
                m = yc.mean(0)
                S = (yc - m).T @ (yc - m) / (yc.shape[0] - 1)
                v = torch.diagonal(S)
                p = v.numel()
                on = torch.ones_like(v) if q in (1, p) else (torch.arange(p, device=v.device) < q).to(v.dtype)
                sg = torch.where(((yc - m) ** 3).mean(0) >= 0, 1.0, -1.0)
                de = on * sg * torch.sqrt(math.pi * (1.0 - al) * v / (math.pi - 2.0))
                P["Sigma"].append(S - (1.0 - al) * torch.diag(v * on))
                P["mu"].append(m - math.sqrt(2.0 / math.pi) * de)
                P["Delta"].append(de[:, None] if q == 1 else torch.diag(de)[:, :q])
                P["pi"].append(torch.tensor(yc.shape[0] / y.shape[0], dtype=y.dtype, device=y.device))
                P["nu"].append(torch.tensor(10.0, dtype=y.dtype, device=y.device))
            yield {k: torch.stack(v) for k, v in P.items()}


def _np(d):
    return {k: v.cpu().numpy() if isinstance(v, torch.Tensor) else v for k, v in d.items()}


def exact(case, seed):
    # what this takes: the evaluations of a normal CDF or of sin^(nu-1) in FP64
    steps = {"fit": case["iters"] + 1, "batch": case["iters"] + 1, "start": 9 * case.get("starts", 1)}.get(case["kind"], 1)
    total = 0.0
    for p, q, g, n in _shapes(case):
        ev = {1: 40.0, 2: 2 * 48 * 40.0}
        ev.update({k: 2.0 * k * N_LATTICE * M_SHIFTS for k in range(3, 9)})
        one = ev[q] if case["kind"] in ("score", "start") or (case["moments"] == 1 and q >= 3) else \
            2 * ev[q] + q * ev.get(q - 1, 0.0) + q * (q - 1) * ev.get(q - 2, 0.0)
        total += steps * g * n * one
    if total > 6e10:
        return None
    outs = []
    for f in _inputs(case, seed):
        y, P, mom = _t(f["y"]), {k: _t(v) for k, v in f["params"].items()}, case["moments"]
        if case["kind"] == "score":
            return _np(dict(loglik=_estep(y, P, mom, True)[0][None]))
        if case["kind"] == "start":
            best, table = None, []
            for Q in _starts(y, torch.as_tensor(f["labels"], device=y.device), f["g"], f["q"]):
                ok = all(torch.linalg.cholesky_ex(Q["Sigma"][h])[1] == 0 for h in range(f["g"]))
                table.append(float(_estep(y, Q, mom, True)[0]) if ok else -math.inf)
                if best is None or table[-1] > table[best[0]]:
                    best = (len(table) - 1, Q)
            return _np(dict(best[1], table=np.array(table).reshape(case["starts"], 9), best=np.array([best[0]])))
        if case["kind"] in ("fit", "batch"):
            hist = []
            for _ in range(case["iters"]):
                L, E = _estep(y, P, mom)
                hist.append(float(L))
                P = _mstep(_stats(y, P, E), P, f["n"])
            hist.append(float(_estep(y, P, mom, True)[0]))
            outs.append(dict(_np(P), hist=np.array(hist)))
            continue
        L, E = _estep(y, P, mom)
        if case["kind"] == "pairs":  # the standard errors of the lattice have no exact value
            return _np(dict(E, loglik=L[None], se=None))
        S = _stats(y, P, E)
        out = dict(_mstep(S, P, f["n"]), loglik=L[None])
        if case["kind"] == "em":
            out["stats"] = S
        return _np(out)
    if case["kind"] == "fit":
        return dict(outs[0], iters=np.array([case["iters"]]))
    flat = {k: np.concatenate([o[k].ravel() for o in outs]) for k in NAMES}
    n = len(outs)
    return dict(flat, hist=np.stack([o["hist"] for o in outs]), iters=np.full(n, case["iters"], dtype=np.int32),
                status=np.zeros(n, dtype=np.int32))
