"""GPU: the chi tables of the FP32 modes (log s interpolated over the normal score of the lattice's
first coordinate), where they can go wrong: dofs near 1 and large ones (Newton's two starts), both
tails, few points and many points (the table's range follows the points).

Against the FP64 mode, whose tables hold the quantiles themselves, on the same points, at the
documented FP32 tolerances: log f within 3 standard errors + 5e-5, u 1e-4.
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


@pytest.mark.parametrize("nu", [0.3, 2.5, 60.0, 4000.0, 3e4])
@pytest.mark.parametrize("npoints,nshifts", [(33, 2), (1024, 8), (16411, 2)])
def test_chi_tables(cf, nu, npoints, nshifts):
    q, n = 3, 6
    rng = np.random.default_rng(31)
    par = synth.draw_params(rng, q, q, 1, wishart_df=2 * q + 4, delta_sd=0.5)
    y, _ = synth.sample(rng, n, par)
    par["nu"] = np.array([nu])
    out = []
    for prec in (0, 1):
        ctx = cf.cfust_create(q, q, 1, n, cf.cfust_default_opts(precision=prec, moments=1, qmc_points=npoints,
                                                                qmc_shifts=nshifts, seed=11, nu_min=0.1, nu_max=1e5))
        cf.cfust_set_data(ctx, y)
        cf.cfust_set_params(ctx, par)
        cf.cfust_estep(ctx)
        alpha_s = cf.cfust_debug_read(ctx, 6)[:n].reshape(1, n)
        out.append((cf.cfust_get_pairs(ctx), alpha_s))
    (ref, al), (got, _) = out
    se = 3.0 * ref["se"] / al
    err = np.abs(got["logf"] - ref["logf"])
    err_u = np.abs(got["u"] / ref["u"] - 1.0)
    print(f"nu={nu} N={npoints}: logf {err.max():.1e} u {err_u.max():.1e}")
    assert (err <= se + 5e-5).all()
    assert err_u.max() <= 1e-4
