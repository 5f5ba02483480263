"""GPU: pairs sent to the FP64 fix-up of which one limit is exactly 0 (an observation at the
location in one coordinate): Phi(0) at every lattice point.  Against the FP64 form at the
tolerances of the far-tail test: log f 1e-12, u 1e-10, the single pass's moments 1e-9 of their largest value.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("moments", [0, 1])
def test_zero_limit(moments):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1606_02054_gb300 as cf

    p = 3
    y = np.array([[-1.0, 0.0, 0.0], [0.0, -1.25, 0.0], [0.0, 0.0, -1.5], [-1.0, 0.0, 0.5], [1.0, 0.5, 0.0]])
    par = dict(pi=np.ones(1), mu=np.zeros((1, p)), Sigma=1e-3 * np.eye(p)[None], Delta=np.eye(p)[None], nu=np.array([30.0]))
    got = []
    for precision in (cf.CFUST_PREC_FP64, cf.CFUST_PREC_FP32):
        ctx = cf.cfust_create(p, p, 1, len(y), cf.cfust_default_opts(precision=precision, moments=moments, qmc_points=256,
                                                                     qmc_shifts=4))
        cf.cfust_set_data(ctx, y)
        cf.cfust_set_params(ctx, par)
        cf.cfust_estep(ctx)
        got.append({k: v[0][:4] for k, v in cf.cfust_get_pairs(ctx).items() if k != "se"})
    f64, f32 = got
    assert np.all(f64["logf"] < -75.0)  # alpha_s far below 1e-35: all four are listed
    checks = [("logf", 1e-12 * np.abs(f64["logf"])), ("u", 1e-10 * f64["u"])]
    if moments:  # the recursion's moments cancel to nothing this far out, in every form
        checks += [(k, 1e-9 * np.abs(f64[k]).max()) for k in ("eu", "euu")]
    for k, tol in checks:
        print(k, np.abs(f32[k] - f64[k]).max())
        assert np.all(np.abs(f32[k] - f64[k]) <= tol), k
