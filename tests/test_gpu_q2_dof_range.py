"""GPU: FP64 E-steps over the whole range of dofs that a context accepts, where the per-dof
tables of T_1 and T_2 end (internal.cuh, H1_DOF_MAX = 250): moments and M-step of components
whose level-1 dof nu + p + 1 lies below and above that limit, nu stepping across it between two
E-steps, against the oracle; and components in the normal limit nu = infinity beside finite ones; and T_2
down to the end of the FP64 range.

Tolerances: those of the parity tests: log f 1e-9, u 1e-8, the moments 1e-7 of the row scale (the
recursion's formulas cancel in the far tails), one M-step 1e-8; log-likelihood of the FP32 and mixed
forms 1e-6.
"""
import numpy as np
import pytest
import scipy.stats

from paper_1606_02054_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cf():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1606_02054_gb300 import build

    build.build()
    import paper_1606_02054_gb300 as cf

    return cf


def _inputs(p, q, n, nu):
    rng = np.random.default_rng(17 * p + n)
    par = synth.draw_params(rng, p, q, len(nu), delta_sd=0.8)
    par["pi"] = np.full(len(nu), 1.0 / len(nu))
    par["nu"] = np.asarray(nu, dtype=float)
    y, _ = synth.sample(rng, n, dict(par, nu=np.minimum(par["nu"], 200.0)))
    return y, par


def _ctx(cf, y, par, nu_max=6000.0, precision=0):
    p, q = par["Delta"].shape[1:]
    qs = synth.qmc_settings(2, npoints=256, nshifts=4)
    ctx = cf.cfust_create(p, q, len(par["nu"]), len(y), cf.cfust_default_opts(
        precision=precision, qmc_points=qs["npoints"], qmc_shifts=qs["nshifts"], qmc_korobov_a=qs["korobov_a"],
        seed=qs["seed"], nu_max=nu_max, hold=cf.CFUST_HOLD_NU))
    cf.cfust_set_data(ctx, y)
    cf.cfust_set_params(ctx, par)
    return ctx, qs


def _check_pairs(got, o):
    live = np.isfinite(o["logf"])
    err = np.abs(got["logf"] - o["logf"])[live] / np.maximum(1.0, np.abs(o["logf"][live]))
    print(f"log f worst {err.max():.2e}, u {np.max(np.abs(got['u'] / o['u'] - 1.0)[live]):.2e}")
    assert err.max() <= 1e-9
    assert np.all(np.abs(got["u"] - o["u"])[live] <= 1e-8 * o["u"][live] + 1e-12)
    for k, axis in (("eu", -1), ("euu", (-2, -1))):
        scale = np.abs(o[k]).max(axis=axis, keepdims=True)
        err = np.abs(got[k] - o[k])[live] / (scale[live] + 1e-3)
        print(f"{k} worst {err.max():.2e} of the row scale")
        assert err.max() <= 1e-7


# nu + p + 1 = 249, 253, 255, 400; the first E-step fills every table from smaller dofs
@pytest.mark.parametrize("p", [2, 5])
def test_moments_across_the_table_limit(cf, oracle, p):
    nu = np.array([249.0, 253.0, 255.0, 400.0]) - p - 1
    y, par = _inputs(p, 2, 61, nu)
    ctx, qs = _ctx(cf, y, dict(par, nu=np.array([30.0, 60.0, 5.0, 200.0])))
    cf.cfust_estep(ctx)
    cf.cfust_set_params(ctx, par)
    L = cf.cfust_estep(ctx)
    got = cf.cfust_get_pairs(ctx)
    o = oracle.estep(y, par, oracle.qmc(**qs))
    assert abs(L - o["loglik"]) <= 1e-9 * abs(o["loglik"])
    _check_pairs(got, o)
    fresh, _ = _ctx(cf, y, par)
    assert cf.cfust_estep(fresh) == L
    again = cf.cfust_get_pairs(fresh)
    for k in ("logf", "u", "elogu", "eu", "euu", "tau"):
        assert np.array_equal(got[k], again[k]), k
    cf.cfust_mstep(ctx)
    new = cf.cfust_get_params(ctx)
    ref, _ = oracle.mstep(y, o, par, nu_max=6000.0, hold=oracle.HOLD_NU)
    for k in ("pi", "mu", "Sigma", "Delta", "nu"):
        assert np.allclose(new[k], ref[k], rtol=1e-8, atol=1e-10), k


# one component with the normal limit beside one with a finite nu (nu_max = infinity): the level-0
# T_2 at q = 2, the level-1 and level-2 ones at q = 3 and 4
@pytest.mark.parametrize("p,q,precision", [(2, 2, 0), (4, 2, 0), (3, 3, 0), (4, 4, 0), (2, 2, 1), (2, 2, 2)])
def test_infinite_nu(cf, oracle, p, q, precision):
    y, par = _inputs(p, q, 41, (np.inf, 7.0))
    if precision == 2:
        y = y.astype(np.float32)
    ctx, qs = _ctx(cf, y, par, nu_max=np.inf, precision=precision)
    L = cf.cfust_estep(ctx)
    got = cf.cfust_get_pairs(ctx)
    o = oracle.estep(y.astype(np.float64), par, oracle.qmc(**qs))
    assert abs(L - o["loglik"]) <= (1e-6 if precision else 1e-9) * abs(o["loglik"])
    assert abs(cf.cfust_loglik(ctx) - o["loglik"]) <= (1e-6 if precision else 1e-9) * abs(o["loglik"])
    if not precision:
        _check_pairs(got, o)
    assert np.all(got["u"][0] == 1.0)


def test_smallest_t2(cf, oracle):
    """T_2 between 1e-307 and 1e-290 (the FP64 range ends at 2e-308): log f, u and the moments
    as elsewhere, no null pair."""
    p = q = 2
    par = dict(pi=np.ones(1), mu=np.zeros((1, p)), Sigma=1e-3 * np.eye(p)[None],
               Delta=np.array([[[1.0, 0.2], [0.3, 1.0]]]), nu=np.array([190.0]))
    ray = np.concatenate([np.geomspace(5.0, 1e3, 120)[:, None] * np.array([[-1.0, -a]]) for a in (1.0, 0.98)])
    o = oracle.estep(ray, par, oracle.qmc())
    Om = par["Sigma"][0] + par["Delta"][0] @ par["Delta"][0].T
    logtp = scipy.stats.multivariate_t(shape=Om, df=190.0).logpdf(ray)
    log10 = (o["logf"][0] - logtp - 2.0 * np.log(2.0)) / np.log(10.0)
    keep = (log10 > -307.0) & (log10 < -290.0)
    assert keep.sum() >= 20 and np.sum(log10[keep] < -301.0) >= 5, log10
    y = ray[keep]
    ctx, qs = _ctx(cf, y, par)
    L = cf.cfust_estep(ctx)
    got = cf.cfust_get_pairs(ctx)
    o = oracle.estep(y, par, oracle.qmc(**qs))
    assert np.isfinite(L) and np.all(np.isfinite(got["logf"]))
    _check_pairs(got, o)
    # subnormal T_2: no null pair, no overflow of 1/T_2
    y = ray[(log10 > -310.0) & (log10 < -308.0)]
    assert len(y) >= 5
    ctx, _ = _ctx(cf, y, par)
    assert np.isfinite(cf.cfust_estep(ctx))
    got = cf.cfust_get_pairs(ctx)
    assert all(np.all(np.isfinite(got[k])) for k in ("logf", "u", "elogu", "eu", "euu"))
