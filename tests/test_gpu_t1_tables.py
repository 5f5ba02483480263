"""GPU: FP64 T_1 and T_2 through the per-dof tables (internal.cuh, H1_*), where they can go
wrong: the lowest dofs, the dof limit of the tables crossed within one E-step, rho = 0, |rho|
on both sides of the grading threshold 0.99 with both signs, a record per warp up to full
warps, the T_1 records of q = 1 to 3.

T_2 records (q = 2) against cfust_tk_eval, which takes the continued fraction inside the same
nodes, so that the quadrature's own error (1.8e-9 at |rho| > 0.99 and dof 250) is in neither
side's way.  Tolerance 1e-11 relative: both sides raise a sine to a power of up to 250 through
its logarithm, up to 50 bits long, which rounds to 250 * 50 * ln 2 * 1.1e-16 = 1e-12 at worst
in each of a few factors.  q = 1 and 3 against the oracle at the parity tests' tolerances.
"""
import numpy as np
import pytest

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


def _setup(cf, p, q, n, nu):
    """Components: rho = 0; columns of Delta nearly parallel, then nearly opposite (Lambda's
    correlations near -1 and +1); a drawn one."""
    rng = np.random.default_rng(1000 * p + n)
    g = 4
    par = synth.draw_params(rng, p, q, g, wishart_df=max(8, 2 * p))
    par["pi"] = np.full(g, 0.25)
    par["Sigma"][0] = np.eye(p)
    par["Delta"][0] = np.eye(p, q) * 1.3
    for h, sign in ((1, 1.0), (2, -1.0)):
        col = rng.normal(0.0, 1.5, p)
        par["Sigma"][h] = np.eye(p) * 0.05
        par["Delta"][h] = np.stack([col * (1.0 if k == 0 else sign * (1.0 + 0.02 * k)) for k in range(q)], axis=1)
    par["nu"] = np.asarray(nu, dtype=float)
    y, _ = synth.sample(rng, n, par)
    qs = dict(synth.qmc_settings(), npoints=128, nshifts=4)
    ctx = cf.cfust_create(p, q, g, n, cf.cfust_default_opts(
        qmc_points=qs["npoints"], qmc_shifts=qs["nshifts"], qmc_korobov_a=qs["korobov_a"], seed=qs["seed"],
        nu_max=6000.0))
    cf.cfust_set_data(ctx, y)
    cf.cfust_set_params(ctx, par)
    return ctx, y, par, qs


@pytest.mark.parametrize("p,n,nu", [
    (2, 1, (1.0, 1.5, 2.5, 4.0)),
    (2, 97, (1.0, 1.2, 3.0, 60.0)),
    (2, 97, (246.9, 247.5, 248.2, 290.0)),
    (32, 160, (20.0, 200.0, 217.5, 218.5)),
    (5, 2003, (5.0, 9.0, 30.0, 110.0)),
])
def test_t2_records(cf, p, n, nu):
    q = 2
    ctx, y, par, _ = _setup(cf, p, q, n, nu)
    cf.cfust_estep(ctx)
    bt = cf.cfust_debug_read(ctx, 3).reshape(4, n, 2, q)
    got = cf.cfust_debug_read(ctx, 6).reshape(4, n, 2)
    F = cf.cfust_debug_read(ctx, 0).reshape(4, -1)
    rho = F[:, p + p * p + p * q + 4 + q * q + q + q]  # row 1, column 0 of the correlation factor
    assert rho[0] == 0.0 and rho[1] < -0.9 and rho[2] > 0.9, rho
    V = np.zeros((4, n, 2, q, q))
    V[..., 0, 0] = V[..., 1, 1] = 1.0
    V[..., 0, 1] = V[..., 1, 0] = rho[:, None, None]
    dof = np.zeros((4, n, 2)) + (par["nu"] + p)[:, None, None] + np.array([0.0, 2.0])
    ref, _ = cf.cfust_tk_eval(ctx, bt.reshape(-1, q), V.reshape(-1, q, q), dof.ravel())
    ref = ref.reshape(got.shape)
    err = np.abs(got - ref) / np.maximum(ref, 1e-290)
    print(f"p={p} n={n} nu={nu}: worst {err.max():.2e}, rho {rho}")
    assert err.max() <= 1e-11


@pytest.mark.parametrize("p,q,n,nu", [
    (2, 1, 331, (1.0, 7.0, 180.0, 5000.0)),
    (3, 3, 17, (1.0, 6.0, 60.0, 249.0)),
])
def test_t1_records(cf, oracle, p, q, n, nu):
    ctx, y, par, qs = _setup(cf, p, q, n, nu)
    L = cf.cfust_estep(ctx)
    got = cf.cfust_get_pairs(ctx)
    o = oracle.estep(y, par, oracle.qmc(**qs))
    assert abs(L - o["loglik"]) <= 1e-9 * abs(o["loglik"])
    ok = o["tau"] > 1e-200
    for k, rtol in (("logf", 1e-9), ("u", 1e-9 if q < 3 else 1e-8)):
        err = np.abs(got[k] - o[k])[ok] / np.maximum(1.0 if k == "logf" else 0.0, np.abs(o[k][ok]))
        print(f"p={p} q={q} n={n} {k}: worst {err.max():.2e}")
        assert err.max() <= rtol


@pytest.mark.parametrize("precision,rtol", [(0, 1e-12), (1, 5e-5)])
def test_level1_read_back(cf, oracle, precision, rtol):
    """At q = 2 the E-step forms the level-1 T_1 inside combine; the diagnostic read-back still
    gives their limits and values."""
    ctx, y, par, _ = _setup(cf, 2, 2, 41, (1.0, 6.0, 60.0, 150.0))
    if precision:
        ctx = cf.cfust_create(2, 2, 4, 41, cf.cfust_default_opts(precision=precision))
        cf.cfust_set_data(ctx, y)
        cf.cfust_set_params(ctx, par)
    cf.cfust_estep(ctx)
    before = cf.cfust_debug_read(ctx, 6).copy()
    bt = cf.cfust_debug_read(ctx, 4).reshape(4, 41, 2)
    got = cf.cfust_debug_read(ctx, 7).reshape(4, 41, 2)
    ref = np.array([[[oracle.t1cdf(b, par["nu"][h] + 3) for b in row] for row in bt[h]] for h in range(4)])
    ok = ref > 1e-30  # within FP32's range
    assert ok.mean() > 0.9 and np.abs(got / ref - 1.0)[ok].max() <= rtol
    assert np.array_equal(before, cf.cfust_debug_read(ctx, 6))
