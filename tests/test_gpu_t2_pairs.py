"""GPU: the FP32 T_2 pieces in packed pairs of nodes and the FP32 tables of H, where they can go
wrong: an odd node count (the last pair is padded), dofs beyond the tables' full range (sigma_max
< 1), rho = 0 and |rho| beyond the grading threshold, 1 to 4 records per lane of a chunk.

Values against the FP64 mode at the same node count, so that the quadrature's own error (2e-3 for
steep records at dof 300) is on both sides.  Tolerance: the documented FP32 floor 5e-5, or where the
dof is larger the bound of the two powers' exponents, (dof - 1)/2 ln 2 times the 2^-22 error of the
approximate log2 each.  A record's value does not depend on the chunk it is in, so the chunk
lengths are compared bit for bit.
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


def _records(cf, y, par, precision=1, **kw):
    n, p = y.shape
    g = len(par["nu"])
    ctx = cf.cfust_create(p, 2, g, n, cf.cfust_default_opts(precision=precision, nu_max=6000.0, **kw))
    cf.cfust_set_data(ctx, y)
    cf.cfust_set_params(ctx, par)
    cf.cfust_estep(ctx)
    val = cf.cfust_debug_read(ctx, 6).reshape(g, n, 2)
    F = cf.cfust_debug_read(ctx, 0).reshape(g, -1)
    return val, F[:, p + p * p + p * 2 + 4 + 4 + 2 + 2]  # values, rho per component


def _params(rng, p, nu):
    par = synth.draw_params(rng, p, 2, 4, wishart_df=2 * p + 4)
    par["pi"] = np.full(4, 0.25)
    par["Sigma"][0] = np.eye(p)
    par["Delta"][0] = np.eye(p, 2) * 1.3
    col = rng.normal(0.0, 1.5, p)
    par["Sigma"][1] = np.eye(p) * 0.05
    par["Delta"][1] = np.stack([col, 1.02 * col], axis=1)
    par["nu"] = np.asarray(nu, dtype=float)
    return par


@pytest.mark.parametrize("p,n,nu,t2_nodes", [
    (3, 1, (3.0, 8.0, 20.0, 60.0), 64),
    (3, 67, (3.0, 8.0, 20.0, 60.0), 33),
    (8, 67, (4.0, 9.0, 240.0, 300.0), 64),
    (5, 67, (700.0, 40.0, 1000.0, 2000.0), 64),
])
def test_t2_pairs(cf, p, n, nu, t2_nodes):
    rng = np.random.default_rng(10 * p + n)
    par = _params(rng, p, nu)
    y, _ = synth.sample(rng, n, par)
    val, rho = _records(cf, y, par, t2_nodes=t2_nodes)
    ref, _ = _records(cf, y, par, precision=0, t2_nodes=t2_nodes)
    assert rho[0] == 0.0 and rho[1] < -0.9
    dof = (par["nu"] + p)[:, None, None] + np.array([0.0, 2.0])
    tol = np.maximum(5e-5, (dof - 1.0) * np.log(2.0) * 2.0 ** -22)
    ok = ref > 1e-25
    if t2_nodes != 64:  # graded pieces have 64 nodes in FP32
        ok &= (np.abs(rho) < 0.99)[:, None, None]
    err = np.where(ok, np.abs(val / np.maximum(ref, 1e-25) - 1.0), 0.0)
    print(f"p={p} n={n} nu={nu} t2_nodes={t2_nodes}: worst {err.max():.2e} ({(err / tol).max():.2f} of the bound)")
    assert (err <= tol).all()


@pytest.mark.parametrize("n", [20_000, 30_000, 50_001])
def test_t2_chunk_lengths(cf, n):
    rng = np.random.default_rng(3)
    par = _params(rng, 4, (3.0, 8.0, 20.0, 60.0))
    y, _ = synth.sample(rng, n, par)
    val, _ = _records(cf, y, par)  # 8 n records: 2, 2 and 3 per lane
    sub = np.concatenate([np.arange(150), np.arange(n - 150, n)])
    few, _ = _records(cf, y[sub], par)  # 1 per lane
    assert np.array_equal(val[:, sub], few)
