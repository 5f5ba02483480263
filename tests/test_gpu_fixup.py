"""GPU: the FP64 fix-up of far-tail pairs in the FP32 modes (alpha_s below 1e-35), cut into tasks
(short lists) and with a warp per pair (lists longer than FIX_CAP = 1024), against the FP64
mode on the same points.

Tolerances: both sides sum the same points in FP64; as in the parity tests at q >= 3, 1e-8 on
log f and u and 1e-7 of the row scale on eu (q = 2: 1e-8 on log f, the deterministic T_2).  The mixed
form whitens in FP32 before the list is made, but the fix-up whitens in FP64: the same bounds, its
rows stored in FP32 (2e-7 more).
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


def _problem(p, q, n_far, seed):
    """Component 0 holds the body; component 1 is skewed away from every observation of the
    far group, whose pairs with it have alpha_s far below FP32's range."""
    rng = np.random.default_rng(seed)
    par = synth.draw_params(rng, p, q, 2, nu_range=(8.0, 9.0))
    par["pi"] = np.array([0.9, 0.1])
    par["mu"] = np.stack([np.full(p, -9.0), np.zeros(p)])
    par["Sigma"] = np.stack([np.eye(p) * 2.0, np.eye(p) * 0.16])
    par["Delta"][0] *= 0.1
    par["Delta"][1] = np.eye(p, q) * (1.2 if p == q else 6.0)
    par["nu"] = np.array([8.0, 199.0])
    far = -9.0 + 1.5 * rng.standard_normal((n_far, p))
    near = np.abs(rng.standard_normal((37, p)))
    return np.concatenate([far, near]), par


@pytest.mark.parametrize("p,q,n_far,precision,moments,npoints,nshifts", [
    (3, 3, 5, 1, 1, 1024, 8),
    (4, 4, 40, 1, 0, 512, 4),
    (5, 3, 61, 2, 1, 1000, 7),
    (6, 6, 9, 2, 1, 96, 64),
    (2, 2, 33, 1, 0, 64, 2),
    (3, 3, 1500, 1, 1, 64, 4),
    (3, 3, 1300, 2, 1, 64, 4),
])
def test_fixup(cf, p, q, n_far, precision, moments, npoints, nshifts):
    y, par = _problem(p, q, n_far, 17 * q + n_far)
    n = y.shape[0]

    def ctx(prec):
        c = cf.cfust_create(p, q, 2, n, cf.cfust_default_opts(precision=prec, moments=moments, qmc_points=npoints,
                                                              qmc_shifts=nshifts, seed=5))
        cf.cfust_set_data(c, y)
        cf.cfust_set_params(c, par)
        return c

    ref_c, c = ctx(0), ctx(precision)
    ref_L = cf.cfust_estep(ref_c)
    ref = cf.cfust_get_pairs(ref_c)
    m0 = 1 if moments == 1 and q >= 3 else 2
    alpha_s = cf.cfust_debug_read(ref_c, 6)[:2 * n * m0].reshape(2, n, m0)[..., 0]
    far = (alpha_s < 1e-36) & (alpha_s > 1e-280)
    assert far.sum() >= min(n_far, 1100 if n_far > 1024 else n_far) * 0.8, far.sum()
    for _ in range(2):  # the second E-step reuses the task buffers
        L = cf.cfust_estep(c)
        got = cf.cfust_get_pairs(c)
        assert abs(L - ref_L) <= 5e-5 * n  # the other pairs' FP32 floor
        extra = 2e-7 if precision == 2 else 0.0
        err = np.abs(got["logf"] - ref["logf"])[far] / np.abs(ref["logf"][far])
        print(f"q={q} far={far.sum()} logf {err.max():.2e}")
        assert err.max() <= 1e-8
        if q >= 3:
            err = np.abs(got["u"] / ref["u"] - 1.0)[far]
            scale = np.abs(ref["eu"][far]).max(axis=1, keepdims=True)
            err_eu = np.abs(got["eu"] - ref["eu"])[far] / scale
            print(f"   u {err.max():.2e} eu {err_eu.max():.2e}")
            assert err.max() <= 1e-8 + extra
            if moments == 1:  # the recursion's moments cancel this far out
                assert err_eu.max() <= 1e-7 + extra
    dens = cf.cfust_loglik(c)  # the density pass's tasks
    assert abs(dens - cf.cfust_loglik(ref_c)) <= 5e-5 * n
