"""GPU: device functions of csrc/special.cuh that the integrators use in packed or tabulated form,
each evaluated on its own through a small library built from the header here.

Bounds:
  cf_atan2_f32: 2 ulp (the quotient with its remainder 0.5, the series' last operation 0.5, the
      octant's addition 0.5, the fit 0.13); sqrt_newton, rcp_newton: 0.6 ulp (a Newton step on an
      approximation good to 2^-22 leaves 2^-44 before the last rounding; sqrt's remainder is 2^-23 of
      x and has its own 24 bits from x = 2^-100 on).
  h1_eval, h32_eval: exact but for the argument's rounding on tables of a linear function.
  the packed Phi and Phi^-1: those of the scalar forms, whose constants they share
      (tests/test_gpu_special.py); Phi^-1 of p > 1/2 rounds 1 - p once more: 2^-24 over the density there.
  node_log: half an ulp each for the table's entry, the series' sum and the last addition: 3e-16 of
      |log v|, and 1e-18 where v is near 1 (entries below 2^-7); node_exp: the reduction, the
      series and the product: 4e-16 relative; the whole range of exp() with FAR.
  ncdf_tab: the exponential, the polynomial and two products: 1e-15 relative; ncdfinv_tab: 1e-15 of
      max(1, |y|) (the quotient and the difference of Mills ratios of at most 1/2, times sqrt(2 pi)).
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import scipy.special as sp

pytestmark = pytest.mark.gpu

SRC = r"""
#include "internal.cuh"
#include "special.cuh"
__global__ void f32_kernel(int fn, int n, const float* x, const float* y, float* out)
{
    for (int i = 2 * (blockIdx.x * blockDim.x + threadIdx.x); i < n; i += 2 * gridDim.x * blockDim.x) {
        if (fn < 3) {  // packed pairs
            f32x2 r;
            if (fn == 0) r = ncdf2_signed(pk2(x[i] * NCDF_SCALE, x[i + 1] * NCDF_SCALE));
            else if (fn == 1) r = ncdfinv2_abs(pk2(x[i], x[i + 1]));
            else r = sin2_signed(pk2(x[i], x[i + 1]));
            up2(r, out[i], out[i + 1]);
        } else {
            for (int k = i; k < i + 2; ++k)
                out[k] = fn == 3 ? h32_eval(x[k], reinterpret_cast<const float4*>(y), (float)H32_CELLS)  // y: the table
                       : fn == 4 ? cf_atan2_f32(y[k], x[k]) : fn == 5 ? sqrt_newton(x[k]) : rcp_newton(x[k]);
        }
    }
}
__global__ void __launch_bounds__(128) f64_kernel(int fn, int n, const double* x, const double* tab, double* out)
{
    __shared__ NcdfTables q;
    __shared__ double scratch[(NCDF_CELLS + 4) * H1_NC];
    ncdf_tables_init(q, scratch);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        out[i] = fn == 0 ? ncdf_tab(x[i], q) : fn == 1 ? ncdfinv_tab(x[i], q) 
               : fn == 2 ? h1_eval(x[i], tab) : fn == 3 ? node_log(x[i], q.nt) : node_exp<true>(x[i], q.nt);
}
template <typename T> static T* up(const T* h, int n)
{
    T* d = nullptr;
    if (cudaMalloc(&d, n * sizeof(T)) != cudaSuccess) return nullptr;
    cudaMemcpy(d, h, n * sizeof(T), cudaMemcpyHostToDevice);
    return d;
}
template <typename T> static int down(T* h, T* d, int n) { return (int)cudaMemcpy(h, d, n * sizeof(T), cudaMemcpyDeviceToHost); }
extern "C" int run_f32(int fn, int n, const float* x, int ny, const float* y, float* out)
{
    float *dx = up(x, n), *dy = up(y, ny), *dz = up(out, n);
    if (!dx || !dy || !dz) return -1;
    f32_kernel<<<256, 128>>>(fn, n, dx, dy, dz);
    const int e = down(out, dz, n);
    cudaFree(dx); cudaFree(dy); cudaFree(dz);
    return e;
}
extern "C" int run_f64(int fn, int n, const double* x, int ny, const double* y, double* out)
{
    double *dx = up(x, n), *dy = up(y, ny), *dz = up(out, n);
    if (!dx || !dy || !dz) return -1;
    f64_kernel<<<64, 128>>>(fn, n, dx, dy, dz);
    const int e = down(out, dz, n);
    cudaFree(dx); cudaFree(dy); cudaFree(dz);
    return e;
}
"""


@pytest.fixture(scope="module")
def dev(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1606_02054_gb300 import build as b

    d = tmp_path_factory.mktemp("device_functions")
    src, so = os.path.join(d, "f.cu"), os.path.join(d, "f.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([b._nvcc(), *b.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", b.CSRC, "-I",
                    os.path.join(b.ROOT, "include"), "-o", so, src], check=True)
    lib = ctypes.CDLL(so)

    def run(fn, x, y=None):
        out, y = np.zeros(x.size, x.dtype), x if y is None else np.ascontiguousarray(y, x.dtype)
        assert x.size % 2 == 0
        f = lib.run_f32 if x.dtype == np.float32 else lib.run_f64
        ptr = [v.ctypes.data_as(ctypes.c_void_p) for v in (x, y, out)]
        assert f(fn, x.size, ptr[0], y.size, ptr[1], ptr[2]) == 0
        return out

    return run


def _ulps(got, ref):
    ref32 = np.abs(ref).astype(np.float32)
    return np.abs(got.astype(np.float64) - ref) / (np.nextafter(ref32, np.float32(np.inf)) - ref32).astype(np.float64)


def test_atan2_f32(dev):
    rng = np.random.default_rng(1)
    th, m = rng.uniform(-np.pi, np.pi, 1_000_000), np.exp(rng.uniform(-20.0, 20.0, 1_000_000))
    y, x = (m * np.sin(th)).astype(np.float32), (m * np.cos(th)).astype(np.float32)
    e = _ulps(dev(4, x, y), np.arctan2(y.astype(np.float64), x.astype(np.float64)))
    print(f"atan2: worst {e.max():.2f} ulp, rms {np.sqrt(np.mean(e * e)):.3f}")
    assert e.max() <= 2.0
    big, inf = 3e38, np.inf
    x = np.array([0, 0, 0, 1, -1, big, -big, inf, -inf, 3, -3, big], np.float32)
    y = np.array([0, 1, -1, 0, 0, 1, 1, 2, 2, inf, -inf, big], np.float32)
    # beyond 2^126 the quotient counts as 0 (no angle of that size occurs)
    ref = np.arctan2(y.astype(np.float64), x.astype(np.float64))
    assert np.all(np.abs(dev(4, x, y) - ref)[:-1] <= 3e-7)


def test_newton_f32(dev):
    x = (2.0 ** np.random.default_rng(2).uniform(-100.0, 100.0, 1_000_000)).astype(np.float32)
    assert _ulps(dev(5, x), np.sqrt(x.astype(np.float64))).max() <= 0.6
    assert _ulps(dev(6, x), 1.0 / x.astype(np.float64)).max() <= 0.6


def test_table_lookup(dev):
    """Tables of 64 sigma - 1/2 (FP64, 64 cells) and 256 sigma - 1/2 (FP32, 256): the cells' edges, both ends."""
    s = np.concatenate([np.linspace(0.0, 1.0, 65), np.nextafter(np.linspace(0.0, 1.0, 65)[1:], 0.0),
                        np.random.default_rng(5).uniform(0.0, 1.0, 997), [0.0, 1.0, 1.0 + 2.0 ** -52, 1.0 - 1e-9]])
    tab = np.zeros((64, 10))
    tab[:, 0], tab[:, 1] = np.arange(64), 1.0
    assert np.abs(dev(2, s, tab) - (64.0 * s - 0.5)).max() <= 1e-13
    s = np.concatenate([np.linspace(0.0, 1.0, 257), np.random.default_rng(6).uniform(0.0, 1.0, 999),
                        [1.0 - 2.0 ** -24, 1.0]]).astype(np.float32)
    tab = np.zeros((256, 4))
    tab[:, 0], tab[:, 1] = np.arange(256), 1.0
    assert np.abs(dev(3, s, tab) - (256.0 * s.astype(np.float64) - 0.5)).max() <= 4e-5  # 2 ulp of 256


def test_packed_phi(dev):
    a = np.linspace(-13.0, 9.0, 1_000_000).astype(np.float32)
    got = dev(0, a)
    assert np.all((got < 0) == (a > 0))  # the sign says which side
    rel = np.abs(np.abs(got.astype(np.float64)) / sp.ndtr(a.astype(np.float64)) - 1.0)
    print(f"packed Phi: {rel[a >= -5].max():.2e} (a >= -5), {rel.max():.2e}")
    assert rel[a >= -5].max() <= 4e-6 and rel.max() <= 3e-5


def test_packed_phi_inverse(dev):
    p = np.concatenate([np.logspace(-37, np.log10(0.5), 500_000), np.linspace(0.5, 1.0 - 2.0 ** -24, 500_000)])
    p = np.clip(p.astype(np.float32), np.float32(1e-37), np.float32(1.0 - 2.0 ** -24))
    ref = sp.ndtri(p.astype(np.float64))
    for sign in (1.0, -1.0):
        err = np.abs(dev(1, np.float32(sign) * p) - ref)
        small = np.abs(ref) <= 1
        print(f"packed Phi^-1: {err[small].max():.2e}, {(err[~small] / np.abs(ref[~small])).max():.2e}")
        assert err[small].max() <= 1e-6 and (err[~small] / np.abs(ref[~small])).max() <= 3e-6
    assert np.all(dev(1, np.array([0.0, 1e-38], np.float32)) == dev(1, np.array([1e-37, 1e-37], np.float32)))


def test_packed_sine(dev):
    x = np.linspace(-np.pi, np.pi, 1_000_000).astype(np.float32)
    x = np.clip(x, np.float32(-3.1415925), np.float32(3.1415925))
    err = np.abs(np.abs(dev(2, x).astype(np.float64)) - np.abs(np.sin(x.astype(np.float64))))
    print(f"packed sine: {err.max():.2e}")
    assert err.max() <= 2.5e-7  # the fit 7e-8, the folded angle and the product 1.2e-7


def test_node_functions(dev):
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 120
    rng = np.random.default_rng(3)
    v = np.concatenate([np.exp(rng.uniform(-700.0, 5.0, 1500)), 1.0 + rng.uniform(-0.5, 0.5, 1500),
                        1.0 + np.exp(rng.uniform(-40.0, -1.0, 500)), 1.0 - np.exp(rng.uniform(-36.0, -1.0, 500))])
    ref = [mp.log(mp.mpf(float(t))) for t in v]
    err = np.array([abs(float(mp.mpf(float(g)) - r)) for g, r in zip(dev(3, v), ref)])
    lim = 3e-16 * np.abs(np.array([float(r) for r in ref])) + 1e-18
    print(f"node_log: {np.max(err / lim):.2f} of the bound")
    assert np.all(err <= lim)
    x = np.concatenate([-rng.uniform(0.0, 708.0, 3000), -np.exp(rng.uniform(-40.0, 3.0, 1000)), [0.0, -689.9999, -690.0, -690.0001]])
    ref = [mp.exp(mp.mpf(float(t))) for t in x]
    err = np.array([abs(float(mp.mpf(float(g)) / r - 1)) for g, r in zip(dev(4, x), ref)])
    print(f"node_exp: worst {err.max():.2e}")
    assert err.max() <= 4e-16
    far = dev(4, np.array([-709.5, -740.0, -746.0, -1e300, -np.inf, np.nan]))
    assert np.allclose(far[:2], np.exp([-709.5, -740.0]), rtol=1e-12, atol=5e-324)
    assert np.all(far[2:5] == 0.0) and np.isnan(far[5])


def test_tabulated_phi(dev):
    mp = pytest.importorskip("mpmath")
    mp.mp.prec = 150
    rng = np.random.default_rng(4)
    a = np.concatenate([rng.uniform(-37.0, 8.0, 3000), rng.uniform(-1.0, 1.0, 1000), [0.0, -0.0, 1e-17, -1e-17, 9.0, 40.0]])
    ref = [mp.ncdf(mp.mpf(float(t))) for t in a]
    err = np.array([abs(float(mp.mpf(float(g)) / r - 1)) for g, r in zip(dev(0, a), ref)])
    print(f"ncdf_tab: worst {err.max():.2e}")
    assert err.max() <= 1e-15
    p = np.concatenate([10.0 ** rng.uniform(-300.0, np.log10(0.5), 2000), 1.0 - 10.0 ** rng.uniform(-15.9, np.log10(0.5), 1000),
                        rng.uniform(0.0, 1.0, 1000), [0.25, 0.5, 1e-300, 1.0 - 2.0 ** -53]])
    got = dev(1, p)
    err = []
    for t, g in zip(p, got):  # one Newton step from the value itself: the distance to the root
        y = mp.mpf(float(g))
        tail = mp.ncdf(y) - mp.mpf(float(t)) if y < 0 else (1 - mp.mpf(float(t))) - mp.ncdf(-y)
        err.append(abs(float(tail / mp.npdf(y))) / max(1.0, abs(float(y))))
    print(f"ncdfinv_tab: worst {max(err):.2e} of max(1, |y|)")
    assert max(err) <= 1e-15
