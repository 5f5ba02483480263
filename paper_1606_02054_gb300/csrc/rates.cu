// rates.cu -- cfust_measure_rates: throughput microbenchmarks of the pipes the
// E-step integrators are bound by, measured on the device the library runs on.
//
// The lattice integrators of T_k (k >= 3) spend their time in per-point
// arithmetic: the normal CDF and its inverse (MUFU rcp/ex2/lg2 plus FP32
// polynomials) and the FP32 FMAs of the separation of variables and of the
// moment sums.  No data-sheet number states how fast that mix can run, so it is
// measured here:
//   - FP32 FMA, FP64 FMA: 8 independent FMA chains per thread;
//   - MUFU ex2, lg2, rcp (the approximate PTX forms the FP32 integrators use):
//     8 independent chains per thread;
//   - the single-pass integrand mix of dimension K: per lattice point K normal
//     CDFs, K inverse normal CDFs (this library's packed FP32 forms, ncdf2_signed and
//     ncdfinv2_abs), the K(K-1)/2 + 3K FMAs of the chain and the
//     2 + K + K(K+1)/2 FMAs of the weighted moment sums, with 1 or 2 pairs of
//     points in flight per thread (the better one) and no memory traffic: the
//     rate an implementation of the same algorithm could reach if it did nothing
//     else;
//   - one node of the FP32 T_2 quadrature (two sines, the sin^(nu-1) weight, the
//     inner T_1 through its table), 1 or 2 packed pairs of nodes per thread (the better).
// Every kernel runs a full grid (8 blocks of 256 threads per SM) for a fixed
// number of iterations; rates are operations (or points) per second of
// CUDA-event time after one warm-up launch, and the SM clock is read with
// clock64() against the same events.
#include <cuda_runtime.h>

#include <string>

#include "cfust.h"
#include "internal.cuh"
#include "special.cuh"

void cf_set_global_error(const std::string& msg);

namespace {

constexpr int kThreads = 256;

__global__ void __launch_bounds__(kThreads) fma32_rate_kernel(float* out, int iters, float m, float c)
{
    float a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = threadIdx.x * 1e-7f + k;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
#pragma unroll
            for (int k = 0; k < 8; ++k) a[k] = fmaf(a[k], m, c);
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += a[k];
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

__global__ void __launch_bounds__(kThreads) fma64_rate_kernel(double* out, int iters, double m, double c)
{
    double a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = threadIdx.x * 1e-7 + k;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
#pragma unroll
            for (int k = 0; k < 8; ++k) a[k] = fma(a[k], m, c);
    }
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += a[k];
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

// fn 0: x = ex2(-x) (stays in [0.5, 1]); 1: x = lg2(x) + 1.5 (stays in [0.5, 3]);
// 2: x = rcp(x) + 0.5 (stays near 1.28; the added constant keeps the compiler from
// cancelling two reciprocals)
template <int FN>
__global__ void __launch_bounds__(kThreads) mufu_rate_kernel(float* out, int iters)
{
    float a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = 0.6f + threadIdx.x * 1e-6f + 0.01f * k;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                if constexpr (FN == 0) a[k] = ptx_ex2_approx(-a[k]);
                else if constexpr (FN == 1) a[k] = ptx_lg2_approx(a[k]) + 1.5f;
                else a[k] = ptx_rcp_approx(a[k]) + 0.5f;
            }
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += a[k];
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

// The single-pass integrand of dimension K, packed as mom_pair_f32 computes it (two points in
// the halves of each value), P pairs in flight per thread.  Coordinates w advance by a fixed
// irrational-like step (kept in [0, 1)); the chi variate s is taken from the first coordinate.
template <int K, int P>
__global__ void __launch_bounds__(kThreads) mix_rate_kernel(float* out, int iters)
{
    constexpr int K2 = K * (K + 1) / 2;
    const float t0 = threadIdx.x * (1.0f / 4096.0f);
    f32x2 b[K];
    float nL[K][K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const float v = NCDF_SCALE / (1.0f + 0.05f * r);
        b[r] = pk2((0.3f + 0.1f * r + t0) * v, (0.25f + 0.1f * r + t0) * v);
#pragma unroll
        for (int l = 0; l < K; ++l) nL[r][l] = l < r ? -0.2f / (1 + r + l) * v : 0.f;
    }
    float w[P][K + 1], dw[K + 1];
#pragma unroll
    for (int d = 0; d <= K; ++d) {
        dw[d] = 0.6180339f * (d + 1) - (int)(0.6180339f * (d + 1));
#pragma unroll
        for (int p = 0; p < P; ++p) w[p][d] = 0.5f * dw[d] + 0.125f * p + t0 * 0.1f;
    }
    f32x2 af = 0ull, aw = 0ull, a1[K], a2[K2];
#pragma unroll
    for (int r = 0; r < K; ++r) a1[r] = 0ull;
#pragma unroll
    for (int r = 0; r < K2; ++r) a2[r] = 0ull;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const f32x2 s = pk2(0.5f + w[p][0]);
            f32x2 y[K], f = 0ull;
#pragma unroll
            for (int r = 0; r < K; ++r) {
                f32x2 t = mul2(b[r], s);
#pragma unroll
                for (int l = 0; l < r; ++l) t = fma2(pk2(nL[r][l]), y[l], t);
                const f32x2 e = ncdf2_signed(t);
                f = r == 0 ? e : mul2(f, e);
                y[r] = ncdfinv2_abs(mul2(pk2(w[p][r + 1]), e));
            }
            af = add2(af, f);
            aw = fma2(mul2(f, s), s, aw);
#pragma unroll
            for (int r = 0; r < K; ++r) {
                const f32x2 t = mul2(f, y[r]);
                a1[r] = fma2(t, s, a1[r]);
#pragma unroll
                for (int c = 0; c <= r; ++c) a2[r * (r + 1) / 2 + c] = fma2(t, y[c], a2[r * (r + 1) / 2 + c]);
            }
#pragma unroll
            for (int d = 0; d <= K; ++d) {
                const float t = w[p][d] + dw[d];
                w[p][d] = t >= 1.f ? t - 1.f : t;
            }
        }
    }
    f32x2 s = add2(af, aw);
#pragma unroll
    for (int r = 0; r < K; ++r) s = add2(s, a1[r]);
#pragma unroll
    for (int r = 0; r < K2; ++r) s = add2(s, a2[r]);
    float s0, s1;
    up2(s, s0, s1);
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s0 + s1;
}

// Two neighbouring nodes of the FP32 T_2 quadrature in packed FP32, as t2_pieces_kernel
// computes them: the two sines, the powers (lg2, ex2), the table's cubic and the weighted sum; P
// pairs per thread, angles advancing by a fixed step, the table L1-resident.
template <int P>
__global__ void __launch_bounds__(kThreads) t2node_rate_kernel(float* out, const float4* __restrict__ tab, int iters)
{
    const float t0 = threadIdx.x * (1.0f / 8192.0f);
    f32x2 th[P], acc[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        th[p] = pk2(0.1f + 0.7f * p + t0, 0.4f + 0.7f * p + t0);
        acc[p] = 0ull;
    }
    const float sc = 0.7f, num1 = 7.5f;
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            float D0, D1, s0, s1, e0, e1, g0, g1, u0, u1;
            const f32x2 sp = sin2_signed(th[p]);
            up2(mul2(sp, sp), s0, s1);
            const f32x2 q = mul2(sin2_signed(add2(th[p], pk2(-0.4f))), pk2(sc));
            up2(fma2(q, q, pk2(1.0f)), D0, D1);
            const float r0 = rsqrt_approx(D0), r1 = rsqrt_approx(D1);
            const f32x2 rr = pk2(r0, r1);
            up2(mul2(pk2(ptx_lg2_approx(s0), ptx_lg2_approx(s1)), pk2(0.5f * num1)), e0, e1);
            up2(mul2(pk2(ptx_lg2_approx(D0), ptx_lg2_approx(D1)), pk2(-0.5f * num1)), g0, g1);
            up2(mul2(q & 0x7fffffff7fffffffull, rr), u0, u1);
            const f32x2 H = pk2(h32_eval(u0, tab, (float)H32_CELLS), h32_eval(u1, tab, (float)H32_CELLS));
            const f32x2 T = mul2(mul2(pk2(ptx_ex2_approx(g0), ptx_ex2_approx(g1)), mul2(rr, rr)), H);
            acc[p] = fma2(mul2(pk2(ptx_ex2_approx(e0), ptx_ex2_approx(e1)), T), pk2(0.01f), acc[p]);
            const f32x2 t = add2(th[p], pk2(0.00613f));
            up2(t, u0, u1);
            th[p] = pk2(u0 >= 3.0f ? u0 - 2.9f : u0, u1 >= 3.0f ? u1 - 2.9f : u1);
        }
    }
    float sum = 0.f;
#pragma unroll
    for (int p = 0; p < P; ++p) {
        float a0, a1;
        up2(acc[p], a0, a1);
        sum += a0 + a1;
    }
    out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = sum;
}

__global__ void fill_h32_kernel(float4* tab)
{
    if (threadIdx.x < H32_CELLS) tab[threadIdx.x] = make_float4(0.5f - 0.001f * threadIdx.x, -0.001f, 1e-6f, 1e-9f);
}

__global__ void clock_kernel(long long* out, long long spin)
{
    const long long c0 = clock64();
    while (clock64() - c0 < spin) {
    }
    if (threadIdx.x == 0) out[blockIdx.x] = clock64() - c0;
}

struct Timer {
    cudaEvent_t a = nullptr, b = nullptr;
    cudaError_t init()
    {
        cudaError_t e = cudaEventCreate(&a);
        return e == cudaSuccess ? cudaEventCreate(&b) : e;
    }
    ~Timer()
    {
        if (a) cudaEventDestroy(a);
        if (b) cudaEventDestroy(b);
    }
};

// Launch `launch` once untimed, then once timed; returns seconds.
template <class F>
cudaError_t timed(Timer& t, F launch, double* secs)
{
    launch();
    cudaError_t e = cudaEventRecord(t.a);
    if (e != cudaSuccess) return e;
    launch();
    if ((e = cudaEventRecord(t.b)) != cudaSuccess) return e;
    if ((e = cudaEventSynchronize(t.b)) != cudaSuccess) return e;
    float ms = 0.f;
    if ((e = cudaEventElapsedTime(&ms, t.a, t.b)) != cudaSuccess) return e;
    *secs = ms * 1e-3;
    return cudaGetLastError();
}

// iterations so that one launch takes about `target` seconds, from a first launch of
// `probe` iterations
template <class F>
cudaError_t calibrate(Timer& t, F launch_iters, int probe, double target, int* iters, double* secs)
{
    double s = 0.0;
    cudaError_t e = timed(t, [&] { launch_iters(probe); }, &s);
    if (e != cudaSuccess) return e;
    double scale = s > 0.0 ? target / s : 1.0;
    if (scale > 1e4) scale = 1e4;
    *iters = (int)(probe * scale) > probe ? (int)(probe * scale) : probe;
    return timed(t, [&] { launch_iters(*iters); }, secs);
}

// the better of 1 and 2 independent pairs of points per thread (the rate of the arithmetic alone)
template <int K, int P>
cudaError_t mix_rate_p(Timer& t, float* out, int blocks, double target, double* rate)
{
    int it = 0;
    double s = 0.0;
    cudaError_t e = calibrate(t, [&](int n) { mix_rate_kernel<K, P><<<blocks, kThreads>>>(out, n); }, 64, target, &it, &s);
    if (e == cudaSuccess) {
        const double r = 2.0 * P * blocks * kThreads * it / s;
        if (r > *rate) *rate = r;
    }
    return e;
}

template <int K>
cudaError_t mix_rate(Timer& t, float* out, int blocks, double target, double* rate)
{
    cudaError_t e = mix_rate_p<K, 1>(t, out, blocks, target / 2, rate);
    if (e == cudaSuccess) e = mix_rate_p<K, 2>(t, out, blocks, target / 2, rate);
    return e;
}

template <int P>
cudaError_t t2node_rate(Timer& t, float* out, const float4* tab, int blocks, double target, double* rate)
{
    int it = 0;
    double s = 0.0;
    cudaError_t e = calibrate(t, [&](int n) { t2node_rate_kernel<P><<<blocks, kThreads>>>(out, tab, n); }, 64, target, &it, &s);
    if (e == cudaSuccess) {
        const double r = 2.0 * P * blocks * kThreads * it / s;
        if (r > *rate) *rate = r;
    }
    return e;
}

}  // namespace

extern "C" cfust_status cfust_measure_rates(int device, double seconds, cfust_rates* out)
{
    if (!out || !(seconds > 0.0) || seconds > 5.0) {
        cf_set_global_error("cfust_measure_rates: out is NULL or seconds not in (0, 5]");
        return CFUST_EINVAL;
    }
    *out = cfust_rates{};
    int nsm = 0;
    cudaError_t e = cudaSetDevice(device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) {
        cf_set_global_error(std::string("cfust_measure_rates: ") + cudaGetErrorString(e));
        return CFUST_ECUDA;
    }
    const int blocks = 8 * nsm;
    const size_t nthr = (size_t)blocks * kThreads;
    void* buf = nullptr;
    if ((e = cudaMalloc(&buf, nthr * sizeof(double) + (size_t)nsm * sizeof(long long) +
                                  (H32_CELLS + 1) * sizeof(float4))) != cudaSuccess) {
        cf_set_global_error(std::string("cfust_measure_rates: ") + cudaGetErrorString(e));
        return CFUST_ENOMEM;
    }
    float* f32 = (float*)buf;
    double* f64 = (double*)buf;
    long long* clk = (long long*)((char*)buf + nthr * sizeof(double));
    // behind the clock counts, on a 16-byte boundary
    float4* h32tab = (float4*)((char*)buf + nthr * sizeof(double) + ((size_t)nsm * sizeof(long long) + 15) / 16 * 16);
    Timer t;
    const double tgt = seconds / 13.0;  // 13 measurements share the budget
    int it = 0;
    double s = 0.0;
    do {
        if ((e = t.init()) != cudaSuccess) break;
        // SM clock: cycles counted by clock64() over an event-timed spin of ~tgt
        {
            const long long spin = (long long)(tgt * 1.5e9);
            if ((e = timed(t, [&] { clock_kernel<<<nsm, 32>>>(clk, spin); }, &s)) != cudaSuccess) break;
            long long c = 0;
            if ((e = cudaMemcpy(&c, clk, sizeof(c), cudaMemcpyDeviceToHost)) != cudaSuccess) break;
            out->sm_mhz = (double)c / s / 1e6;
        }
        e = calibrate(t, [&](int n) { fma32_rate_kernel<<<blocks, kThreads>>>(f32, n, 0.9999f, 1e-6f); }, 256, tgt, &it, &s);
        if (e != cudaSuccess) break;
        out->fp32_fma = 128.0 * nthr * it / s;
        e = calibrate(t, [&](int n) { fma64_rate_kernel<<<blocks, kThreads>>>(f64, n, 0.9999, 1e-6); }, 4, tgt, &it, &s);
        if (e != cudaSuccess) break;
        out->fp64_fma = 128.0 * nthr * it / s;
        e = calibrate(t, [&](int n) { mufu_rate_kernel<0><<<blocks, kThreads>>>(f32, n); }, 32, tgt, &it, &s);
        if (e != cudaSuccess) break;
        out->mufu_ex2 = 128.0 * nthr * it / s;
        e = calibrate(t, [&](int n) { mufu_rate_kernel<1><<<blocks, kThreads>>>(f32, n); }, 32, tgt, &it, &s);
        if (e != cudaSuccess) break;
        out->mufu_lg2 = 128.0 * nthr * it / s;
        e = calibrate(t, [&](int n) { mufu_rate_kernel<2><<<blocks, kThreads>>>(f32, n); }, 32, tgt, &it, &s);
        if (e != cudaSuccess) break;
        out->mufu_rcp = 128.0 * nthr * it / s;
        if ((e = mix_rate<3>(t, f32, blocks, tgt, &out->mix_points[3])) != cudaSuccess) break;
        if ((e = mix_rate<4>(t, f32, blocks, tgt, &out->mix_points[4])) != cudaSuccess) break;
        if ((e = mix_rate<5>(t, f32, blocks, tgt, &out->mix_points[5])) != cudaSuccess) break;
        if ((e = mix_rate<6>(t, f32, blocks, tgt, &out->mix_points[6])) != cudaSuccess) break;
        if ((e = mix_rate<7>(t, f32, blocks, tgt, &out->mix_points[7])) != cudaSuccess) break;
        if ((e = mix_rate<8>(t, f32, blocks, tgt, &out->mix_points[8])) != cudaSuccess) break;
        fill_h32_kernel<<<1, 256>>>(h32tab);
        if ((e = t2node_rate<1>(t, f32, h32tab, blocks, tgt / 2, &out->t2_nodes)) != cudaSuccess) break;
        if ((e = t2node_rate<2>(t, f32, h32tab, blocks, tgt / 2, &out->t2_nodes)) != cudaSuccess) break;
    } while (0);
    cudaFree(buf);
    if (e != cudaSuccess) {
        cf_set_global_error(std::string("cfust_measure_rates: ") + cudaGetErrorString(e));
        return CFUST_ECUDA;
    }
    return CFUST_OK;
}
