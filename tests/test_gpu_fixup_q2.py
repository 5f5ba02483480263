"""GPU: long lists of the FP64 fix-up at q <= 2 (more pairs than its task buffer holds: a warp
takes a pair and keeps its values in shared memory), and a list around the buffer's size.  Against
the FP64 form with as many quadrature nodes, at the tolerances of the far-tail test: log f
1e-12, u 1e-10; q = 1 and the normal limit (Phi_2) alike.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q,sigma2,model,n", [(2, 1e-3, 0, 3001), (2, 1e-3, 0, 1024), (2, 1e-3, 0, 1025), (1, 1e-4, 0, 2500),
                                              (2, 0.02, 1, 2050)])
@pytest.mark.parametrize("precision", [1, 2])
def test_long_list(precision, q, sigma2, model, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1606_02054_gb300 as cf

    p = 2
    y = np.random.default_rng(n + q).uniform(-2.6, -2.0, size=(n, p)).astype(np.float32)
    y[:, q:] = 0.0  # q = 1: at the location in the other coordinate
    par = dict(pi=np.ones(1), mu=np.zeros((1, p)), Sigma=sigma2 * np.eye(p)[None], Delta=np.eye(p, q)[None],
               nu=np.array([np.inf if model else 30.0]))
    got = []
    for prec in (0, precision):
        ctx = cf.cfust_create(p, q, 1, n, cf.cfust_default_opts(precision=prec, t2_nodes=64, model=model))
        cf.cfust_set_data(ctx, y if prec == 2 else y.astype(np.float64))
        cf.cfust_set_params(ctx, par)
        L = cf.cfust_estep(ctx)
        pairs = {k: v[0] for k, v in cf.cfust_get_pairs(ctx).items()}
        got.append((L, cf.cfust_loglik(ctx), pairs))
    (L0, _, f64), (L1, l1, f32) = got
    assert np.all(np.isfinite(f64["logf"])) and np.all(f64["logf"] < -70.0)  # every pair is listed
    err = np.abs(f32["logf"] / f64["logf"] - 1.0).max(), np.abs(f32["u"] / f64["u"] - 1.0).max()
    print(f"q={q} n={n} model={model}: log f {err[0]:.2e}, u {err[1]:.2e}")
    assert err[0] <= 1e-12 and err[1] <= (1e-10 if precision == 1 else 1e-7)  # the mixed form stores u in FP32
    assert abs(L1 - L0) <= 1e-12 * abs(L0) and abs(l1 - L0) <= 1e-12 * abs(L0)
