"""GPU: the FP32 lattice passes that take two records per warp (moments and plain T_k), where they
can go wrong: one record, an odd number of records, a change of component between a warp's two
records, numbers of points that are no multiple of the warp (or of two warps), more points than
one 8192-point chunk of the coordinates' fractions, every dimension.

Against the FP64 mode on the same points, at the documented FP32 tolerances: log f within
3 standard errors + 5e-5; u 1e-4 and the single pass's eu 2e-4 of the row scale, where the
pair's weight is not negligible (tau > 1e-12).
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


@pytest.mark.parametrize("q,g,n,moments,npoints,nshifts", [
    (3, 1, 1, 1, 1024, 8),
    (3, 3, 5, 1, 33, 3),
    (4, 3, 7, 1, 100, 2),
    (4, 2, 33, 1, 8193, 3),
    (5, 3, 5, 1, 1024, 8),
    (5, 2, 3, 1, 16411, 2),
    (6, 3, 3, 1, 63, 64),
    (7, 2, 3, 1, 1000, 5),
    (8, 2, 2, 1, 1024, 8),
    (3, 3, 5, 0, 33, 3),
    (4, 3, 3, 0, 1024, 8),
    (5, 2, 3, 0, 8200, 2),
    (8, 1, 1, 0, 96, 4),
])
def test_lattice_pairs(cf, q, g, n, moments, npoints, nshifts):
    rng = np.random.default_rng(100 * q + n)
    par = synth.draw_params(rng, q, q, g, wishart_df=2 * q + 4, delta_sd=0.7)
    y, _ = synth.sample(rng, n, par)
    out = []
    for prec in (0, 1):
        ctx = cf.cfust_create(q, q, g, n, cf.cfust_default_opts(precision=prec, moments=moments, qmc_points=npoints,
                                                                qmc_shifts=nshifts, seed=11))
        cf.cfust_set_data(ctx, y)
        cf.cfust_set_params(ctx, par)
        cf.cfust_estep(ctx)
        m0 = 1 if moments == 1 else 2
        alpha_s = cf.cfust_debug_read(ctx, 6)[:g * n * m0].reshape(g, n, m0)[..., 0]
        out.append((cf.cfust_get_pairs(ctx), alpha_s))
    (ref, al), (got, _) = out
    ok = ref["tau"] > 1e-12
    err = np.abs(got["logf"] - ref["logf"])[ok]
    lim = (3.0 * ref["se"] / al + 5e-5)[ok]
    err_u = np.abs(got["u"] / ref["u"] - 1.0)[ok]
    scale = np.abs(ref["eu"]).max(axis=2, keepdims=True)
    err_eu = (np.abs(got["eu"] - ref["eu"]) / scale)[ok]
    print(f"q={q} n={n} N={npoints}: logf {err.max():.1e} u {err_u.max():.1e} eu {err_eu.max():.1e}")
    assert (err <= lim).all()
    assert err_u.max() <= 1e-4
    if moments == 1:
        assert err_eu.max() <= 2e-4
