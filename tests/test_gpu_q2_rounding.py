"""GPU: the mixed form's assembly at q = 2 rounds u (eq 13) no more often than its formula.

Delta = 0, Sigma = I, mu = 0 and observations on a grid of quarters make c = 0, the squared
distances d exact in FP32 and alpha_s, alpha the same numbers for every observation, so
u (nu + d) / (nu + p) varies by the assembly's rounding alone.  Three correctly rounded operations
(two divisions, one product) have errors of at most 2^-24 each, an rms of at most 2^-24 / sqrt 3
if they are spread evenly, together 2^-24.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,nu", [(2, 8.0), (5, 3.0), (16, 21.0)])
def test_u_rounding_mixed(p, nu):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1606_02054_gb300 as cf

    rng = np.random.default_rng(p)
    n = 4001
    y = (rng.integers(-12, 13, size=(n, p)) / 4.0).astype(np.float32)
    ctx = cf.cfust_create(p, 2, 1, n, cf.cfust_default_opts(precision=cf.CFUST_PREC_MIXED))
    cf.cfust_set_data(ctx, y)
    cf.cfust_set_params(ctx, dict(pi=np.ones(1), mu=np.zeros((1, p)), Sigma=np.eye(p)[None], Delta=np.zeros((1, p, 2)),
                                  nu=np.array([nu])))
    cf.cfust_estep(ctx)
    u = cf.cfust_get_pairs(ctx)["u"][0]
    r = u * (nu + np.sum(y.astype(np.float64) ** 2, axis=1)) / (nu + p)
    rms = np.std(r) / np.mean(r)
    print(f"p={p}: rms rounding of u {rms:.2e} (2^-24 = {2.0 ** -24:.2e}), mean {np.mean(r):.8f}")
    assert abs(np.mean(r) - 1.0) <= 1e-5 and rms <= 2.0 ** -24
