// setup.cu -- per-component factors (S0) and the chi table (S1).
//
// S0, one warp per component, FP64 (definitions under eq (4)):
//   Omega = Sigma + Delta Delta^T, L = chol(Omega), Linv = L^{-1},
//   log|Omega|, A = Linv Delta (so c = A^T Linv (y - mu), d = |Linv (y-mu)|^2),
//   Lambda = I - Delta^T Omega^{-1} Delta = I - A^T A,
//   the constant of the log t_p density (eq 3) and psi((nu+p)/2) of eq (15),
//   and for the truncated-t moments the correlation Cholesky factors of
//   Lambda, of its Schur complements at each r, and of theirs at each s.
// S1: s = sqrt(chi2_nu'^{-1}(w_0)/nu') at every (shift, lattice point) for
//   each tabulated dof nu'; independent of the observations.
#include "internal.cuh"
#include "special.cuh"

namespace {

// Cholesky (lower, row-major, n x n); returns false if not positive definite.
__device__ bool chol_dev(int n, const double* A, double* L)
{
    for (int j = 0; j < n; ++j) {
        double s = A[j * n + j];
        for (int k = 0; k < j; ++k) s -= L[j * n + k] * L[j * n + k];
        if (!(s > 0.0)) return false;
        const double dj = sqrt(s);
        L[j * n + j] = dj;
        for (int i = j + 1; i < n; ++i) {
            double t = A[i * n + j];
            for (int k = 0; k < j; ++k) t -= L[i * n + k] * L[j * n + k];
            L[i * n + j] = t / dj;
        }
        for (int i = 0; i < j; ++i) L[i * n + j] = 0.0;
    }
    return true;
}

// Correlation Cholesky and 1/sqrt(diag) of an n x n scale matrix S.
__device__ bool corr_chol_dev(int n, const double* S, double* dsc, double* Lc)
{
    double R[CF_MAXQ * CF_MAXQ];
    for (int i = 0; i < n; ++i) {
        if (!(S[i * n + i] > 0.0)) return false;
        dsc[i] = 1.0 / sqrt(S[i * n + i]);
    }
    for (int i = 0; i < n; ++i)
        for (int j = 0; j < n; ++j) R[i * n + j] = S[i * n + j] * dsc[i] * dsc[j];
    for (int i = 0; i < n; ++i) R[i * n + i] = 1.0;
    return chol_dev(n, R, Lc);
}

// Schur complement of an n x n matrix S at index r: (n-1) x (n-1), and the
// regression coefficients S_{-r,r}/S_rr.
__device__ void schur_dev(int n, const double* S, int r, double* out, double* mvec)
{
    const double srr = S[r * n + r];
    int ii = 0;
    for (int i = 0; i < n; ++i) {
        if (i == r) continue;
        mvec[ii] = S[i * n + r] / srr;
        int jj = 0;
        for (int j = 0; j < n; ++j) {
            if (j == r) continue;
            out[ii * (n - 1) + jj] = S[i * n + j] - S[i * n + r] * S[r * n + j] / srr;
            ++jj;
        }
        ++ii;
    }
}

}  // namespace

__global__ void __launch_bounds__(32) setup_components_kernel(Dims D, Layout Ly, const double* mu,
                                                              const double* Sigma, const double* Delta,
                                                              const double* nu, double* F, int* flags)
{
    // one warp per component (blockIdx.x); lane i owns row i (Cholesky, A) or column i
    // (L^{-1}); every element is summed in the same order as a serial loop would
    __shared__ double W[CF_MAXP * CF_MAXP];
    __shared__ double Li[CF_MAXP * CF_MAXP];
    const int h = blockIdx.x, lane = threadIdx.x;
    if (h >= D.g) return;
    const int p = D.p, q = D.q;
    const double* Sg = Sigma + (size_t)h * p * p;
    const double* Dl = Delta + (size_t)h * p * q;
    double* Fh = F + (size_t)h * Ly.stride;

    for (int i = lane; i < p; i += 32) Fh[Ly.mu + i] = mu[(size_t)h * p + i];
    // Omega = Sigma + Delta Delta^T (lower triangle of W)
    for (int e = lane; e < p * p; e += 32) {
        const int i = e / p, j = e % p;
        if (j > i) continue;
        double s = Sg[i * p + j];
        for (int k = 0; k < q; ++k) s += Dl[i * q + k] * Dl[j * q + k];
        W[i * p + j] = s;
    }
    __syncwarp();
    // L = chol(Omega) in place, column j at step j: lane i >= j forms its row's entry
    double logdet = 0.0;
    for (int j = 0; j < p; ++j) {
        double t = 0.0;
        if (lane >= j && lane < p) {
            t = W[lane * p + j];
            for (int k = 0; k < j; ++k) t -= W[lane * p + k] * W[j * p + k];
        }
        const double sjj = __shfl_sync(0xffffffffu, t, j);
        if (!(sjj > 0.0)) {
            if (lane == 0) atomicOr(flags, KF_NOTPD_OMEGA);
            return;
        }
        const double dj = sqrt(sjj);
        logdet += 2.0 * log(dj);
        __syncwarp();
        if (lane == j) W[j * p + j] = dj;
        else if (lane > j && lane < p) W[lane * p + j] = t / dj;
        __syncwarp();
    }
    // Linv = L^{-1}: lane c forward-substitutes column c
    for (int c = lane; c < p; c += 32)
        for (int i = 0; i < p; ++i) {
            if (i < c) { Li[i * p + c] = 0.0; continue; }
            double s = (i == c) ? 1.0 : 0.0;
            for (int k = c; k < i; ++k) s -= W[i * p + k] * Li[k * p + c];
            Li[i * p + c] = s / W[i * p + i];
        }
    __syncwarp();
    for (int e = lane; e < p * p; e += 32) Fh[Ly.Linv + e] = Li[e];
    // A = Linv Delta (lane i: row i), into W's upper part is not needed: A goes to Fh and smem
    __shared__ double As[CF_MAXP * CF_MAXQ];
    __shared__ double Lam[CF_MAXQ * CF_MAXQ];
    for (int i = lane; i < p; i += 32)
        for (int k = 0; k < q; ++k) {
            double s = 0.0;
            for (int l = 0; l <= i; ++l) s += Li[i * p + l] * Dl[l * q + k];
            As[i * q + k] = s;
            Fh[Ly.A + i * q + k] = s;
        }
    __syncwarp();
    // Lambda = I - A^T A
    for (int e = lane; e < q * q; e += 32) {
        const int a = e / q, b = e % q;
        double s = (a == b) ? 1.0 : 0.0;
        for (int i = 0; i < p; ++i) s -= As[i * q + a] * As[i * q + b];
        Lam[e] = s;
        Fh[Ly.Lam + e] = s;
    }
    __syncwarp();
    const double v = nu[h];
    if (lane == 0) {
        Fh[Ly.scal + SC_NU] = v;
        if (isinf(v)) {  // nu = infinity: the normal density of eq (2) (CFUSN, eq 5); no eq (15)
            Fh[Ly.scal + SC_LOGTP] = -0.5 * p * log(2.0 * CF_PI) - 0.5 * logdet;
            Fh[Ly.scal + SC_PSI] = 0.0;
        } else {
            Fh[Ly.scal + SC_LOGTP] = lgamma(0.5 * (v + p)) - lgamma(0.5 * v) - 0.5 * p * log(v * CF_PI)
                                   - 0.5 * logdet;
            Fh[Ly.scal + SC_PSI] = cf_digamma(0.5 * (v + p));
        }
        Fh[Ly.scal + SC_RL0] = isinf(v) ? 1.0 : sqrt((v + p + 2.0) / (v + p));
        if (!corr_chol_dev(q, Lam, Fh + Ly.dq, Fh + Ly.Lq)) atomicOr(flags, KF_NOTPD_LAMBDA);
    }
    // level 1: Schur complement of Lambda at each r (lane r), level 2 inside
    const int q1 = q - 1, q2 = q - 2;
    if (lane < q && q1 > 0) {
        const int r = lane;
        double* blk = Fh + Ly.l1 + r * Ly.l1s;
        double* mvec = blk;
        double* sch = blk + q1;
        double* dsc = sch + q1 * q1;
        double* Lc = dsc + q1;
        schur_dev(q, Lam, r, sch, mvec);
        if (!corr_chol_dev(q1, sch, dsc, Lc)) {
            atomicOr(flags, KF_NOTPD_LAMBDA);
            return;
        }
        for (int s2 = 0; s2 < q1 && q2 > 0; ++s2) {
            double* b2 = Fh + Ly.l2 + (r * q1 + s2) * Ly.l2s;
            double sch2[CF_MAXQ * CF_MAXQ];
            schur_dev(q1, sch, s2, sch2, b2);
            if (!corr_chol_dev(q2, sch2, b2 + q2, b2 + 2 * q2)) {
                atomicOr(flags, KF_NOTPD_LAMBDA);
                return;
            }
        }
    }
}

// s = sqrt(chi2_{dof}^{-1}(w_0)/dof) for every dof in `dofs`, shift m and point i.
// Lattice coordinate 0: x = frac(i/N + shift(m, 0)), w = 1 - |2x - 1|.
// rtol: Newton tolerance of the quantile (1e-15 when the FP64 table is used, 1e-9 when only
// the FP32 table is); cst: the per-dof constants (lgamma(dof/2) at CST_LGA).
// Tables k = 0, every, 2 every, ... < ndof (every = 3: only the dof nu+p tables,
// all that the single-pass E-step reads).
__global__ void chi_table_kernel(int ndof, int every, const double* __restrict__ dofs, const double* __restrict__ cst,
                                 Lattice lat, const double* __restrict__ shf, double rtol,
                                 double* __restrict__ t64, float* __restrict__ t32,
                                 double* __restrict__ l64, float* __restrict__ l32)
{
    const long long NM = (long long)lat.M * lat.N;
    const long long total = (long long)((ndof + every - 1) / every) * NM;
    for (long long te = blockIdx.x * (long long)blockDim.x + threadIdx.x; te < total;
         te += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(te % lat.N);
        const int m = (int)((te / lat.N) % lat.M);
        const int k = (int)(te / NM) * every;
        const long long t = k * NM + (te % NM);
        const double dof = dofs[k];
        double x = (double)(((long long)i * lat.z[0]) % lat.N) / (double)lat.N + shf[m * CF_MAXDIM];
        if (x >= 1.0) x -= 1.0;
        const double wc = fabs(2.0 * x - 1.0);
        const double w = 1.0 - wc;
        // dof = infinity (the normal limit): no chi variable, s = 1
        const double x2 = isinf(dof) ? 1.0 : cf_chi2_quantile(w, wc, dof, cst[k * CST_STRIDE + CST_LGA], rtol) / dof;
        const double s = sqrt(x2);
        t64[t] = s;
        t32[t] = (float)s;
        if (l64) {  // log(s^2) (exact E[log W])
            const double ls = log(x2);
            l64[t] = ls;
            l32[t] = (float)ls;
        }
    }
}

// The same tables in the FP32 modes.  The lattice coordinate w_0 of a point never changes, so its
// normal score z = Phi^-1(w_0) is kept (chi_score_kernel, once per context), and log s is a smooth
// function of z (nearly linear for a large dof): degree CHI_D polynomials on CHI_CELLS cells of
// [-zr, zr] through quantiles at the cells' Chebyshev nodes, 320 quantiles a dof instead of
// N x M = 8192.  zr <= 8 covers the lattice's own scores (4.4 at 1024 x 8 points; the extreme
// quantiles are the longest chains); points beyond it take the quantile itself.  Interpolation
// below 3e-14 of s for dof 1 to 1000 at zr = 8 (against scipy; a dof here is nu + p + j > 1), where
// the full table's quantiles were taken to 1e-9 in these modes.  One E-step's tables on a GB300,
// 8192 points, single pass: p = q = g = 4 1.1 -> 0.19 ms, p = q = g = 6 1.4 -> 0.19 ms; what is left
// is a serial chain (a few Newton steps, each an incomplete gamma function).
constexpr int CHI_CELLS = 32, CHI_D = 9, CHI_NC = CHI_D + 1;

__global__ void chi_score_kernel(Lattice lat, const double* __restrict__ shf, double* __restrict__ z)
{
    const int total = lat.M * lat.N;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
        const int i = t % lat.N, m = t / lat.N;
        double x = (double)(((long long)i * lat.z[0]) % lat.N) / (double)lat.N + shf[m * CF_MAXDIM];
        if (x >= 1.0) x -= 1.0;
        const double wc = fabs(2.0 * x - 1.0), w = 1.0 - wc;
        z[t] = w < 0.5 ? normcdfinv(w) : -normcdfinv(wc);
    }
}

// table k = every * blockIdx.x, cell blockIdx.y (a warp of its own: a quantile is a long serial
// chain of FP64 operations, so they are spread over the SMs): the coefficients of log s in powers
// of t in [-1/2, 1/2]
__global__ void __launch_bounds__(32) chi_poly_kernel(int every, double zr, const double* __restrict__ dofs,
                                                      const double* __restrict__ cst, double* __restrict__ coef)
{
    __shared__ double f[CHI_NC], cn[CHI_NC];
    const int k = blockIdx.x * every, cell = blockIdx.y, j = threadIdx.x;
    const double dof = dofs[k];
    if (isinf(dof)) return;  // the normal limit: s = 1
    if (j < CHI_NC) {
        const double z = zr * ((cell + 0.5 + 0.5 * cospi((2 * j + 1) / (2.0 * CHI_NC))) * (2.0 / CHI_CELLS) - 1.0);
        f[j] = 0.5 * log(cf_chi2_node(z, dof, cst[k * CST_STRIDE + CST_LGA]) / dof);
    }
    __syncwarp();
    const double f0 = f[CHI_NC / 2];
    if (j < CHI_NC) {
        double s = 0.0;
        for (int i = 0; i < CHI_NC; ++i) s += (f[i] - f0) * cospi((j * (2 * i + 1) % (4 * CHI_NC)) / (2.0 * CHI_NC));
        cn[j] = s * (j ? 2.0 / CHI_NC : 1.0 / CHI_NC);
    }
    __syncwarp();
    if (j < CHI_NC) {
        double s = 0.0;
        for (int n = CHI_NC - 1; n >= j; --n) s += cn[n] * h1_cheb[n][j];
        s *= (double)(1 << j);  // x = 2 t
        coef[((size_t)k * CHI_CELLS + cell) * CHI_NC + j] = j ? s : s + f0;
    }
}

__global__ void chi_eval_kernel(int ntab, int every, double zr, const double* __restrict__ dofs, const double* __restrict__ cst,
                                Lattice lat, const double* __restrict__ shf, const double* __restrict__ zq,
                                const double* __restrict__ coef, double* __restrict__ t64, float* __restrict__ t32,
                                double* __restrict__ l64, float* __restrict__ l32)
{
    const long long NM = (long long)lat.M * lat.N;
    const long long total = ntab * NM;
    for (long long te = blockIdx.x * (long long)blockDim.x + threadIdx.x; te < total;
         te += (long long)gridDim.x * blockDim.x) {
        const int k = (int)(te / NM) * every;
        const long long at = te % NM, t = k * NM + at;
        const double dof = dofs[k], z = zq[at];
        double ls = 0.0;
        if (!isinf(dof)) {
            if (fabs(z) < zr) {
                const double u = (z + zr) * (0.5 * CHI_CELLS / zr);
                const int c = min((int)u, CHI_CELLS - 1);
                const double x = u - c - 0.5;
                const double* q = coef + ((size_t)k * CHI_CELLS + c) * CHI_NC;
                ls = q[CHI_D];
                for (int i = CHI_D - 1; i >= 0; --i) ls = fma(ls, x, q[i]);
            } else {  // as chi_table_kernel
                const int i = (int)(at % lat.N), m = (int)(at / lat.N);
                double x = (double)(((long long)i * lat.z[0]) % lat.N) / (double)lat.N + shf[m * CF_MAXDIM];
                if (x >= 1.0) x -= 1.0;
                const double wc = fabs(2.0 * x - 1.0);
                ls = 0.5 * log(cf_chi2_quantile(1.0 - wc, wc, dof, cst[k * CST_STRIDE + CST_LGA], 1e-9) / dof);
            }
        }
        const double s = exp(ls);
        t64[t] = s;
        t32[t] = (float)s;
        if (l64) {  // log(s^2) (exact E[log W])
            l64[t] = 2.0 * ls;
            l32[t] = (float)(2.0 * ls);
        }
    }
}

// Degrees of freedom and T_1/T_2 constants for every table index t:
// E-step tables t = 3h + j have dof nu_h + p + j (j = 0: T_q and T_{q-2},
// j = 1: T_{q-1}, j = 2: T_q at nu+p+2); with F == nullptr the dofs are
// already given (cfust_tk_eval, one index per case).
// Four warps share 32 dofs (a lane each), every warp with some of the constants: a constant is a
// serial chain of lgamma, exp and sqrt in FP64, and the kernel is as long as its longest warp.
__global__ void dof_consts_kernel(Dims D, Layout Ly, const double* __restrict__ F, int ndof,
                                  double* dofs, double* c64, float* c32)
{
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, part = warp & 3;
    for (int t = (warp >> 2) * 32 + (threadIdx.x & 31); t < ndof; t += gridDim.x * blockDim.x / 4) {
        double v;
        if (F) {
            const int h = t / 3, j = t % 3;
            v = F[(size_t)h * Ly.stride + Ly.scal + SC_NU] + D.p + j;
            if (part == 0) dofs[t] = v;
        } else {
            v = dofs[t];
        }
        const bool fin = !isinf(v);  // the normal limit uses none of these constants: 0
        auto put = [&](int k, double x) {
            c64[t * CST_STRIDE + k] = x;
            c32[t * CST_STRIDE + k] = (float)x;
        };
        switch (part) {
        case 0:
            put(CST_LGB, fin ? t1_lgb(v) : 0.0);
            put(CST_LGA, fin ? lgamma(0.5 * v) : 0.0);
            break;
        case 1:
            put(CST_LGB1, fin ? t1_lgb(v + 1.0) : 0.0);
            put(CST_C2, fin ? cf_t_const(v) : 0.0);
            break;
        case 2: {
            const double lt = fin ? lgamma(0.5 * (v + 1.0)) - lgamma(0.5 * v) - 0.5 * log(v * CF_PI) : 0.0;
            put(CST_LT1, lt);
            put(CST_ET1, fin ? exp(lt) * sqrt(v) : 0.0);
            break;
        }
        default: {
            const bool ok = fin && v > 1.0;
            const double ltm = ok ? lgamma(0.5 * v) - lgamma(0.5 * (v - 1.0)) - 0.5 * log((v - 1.0) * CF_PI) : 0.0;
            put(CST_LT1M, ltm);
            put(CST_ET1M, ok ? exp(ltm) / sqrt(v - 1.0) : 0.0);
            break;
        }
        }
    }
}

// FP32 observations widened to FP64 (row stride ld).
__global__ void widen_kernel(const float* __restrict__ src, long long ld, Dims D,
                             double* __restrict__ dst)
{
    const long long total = D.n * D.p;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long j = t / D.p;
        const int i = (int)(t % D.p);
        dst[t] = (double)src[j * ld + i];
    }
}

// FP64 observations narrowed to FP32 (mixed precision copy).
__global__ void narrow_kernel(const double* __restrict__ src, Dims D, float* __restrict__ dst)
{
    const long long total = D.n * D.p;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x)
        dst[t] = (float)src[t];
}

// Tables of H for the dofs v = nu_h + p + e (internal.cuh, H1_*): per cell, H at the H1_NC
// Chebyshev nodes (from the continued fraction: with y = 1 - sigma^2 and a = v/2,
// H = sigma C betacf(a, 1/2, y) / v where that one converges fast, else
// 1/2 y^-a - sigma C betacf(1/2, a, sigma^2)), their Chebyshev coefficients and those as powers
// of t in [-1/2, 1/2].  One value of the cell is taken off first, so the sums carry its small
// changes only.  Blocks of 16 cells (blockIdx.x) of table 4h + e (blockIdx.y); a thread per
// node, then per coefficient.
constexpr int H1_TC = 16;  // cells per block
// H(sigma) at dof v, C = cf_t_const(v)
static __device__ double h1_value(double sg, double v, double C)
{
    const double a = 0.5 * v, y = (1.0 - sg) * (1.0 + sg);
    const bool direct = y < (a + 1.0) / (a + 2.5);
    const double cf = betacf_dev<double>(direct ? a : 0.5, direct ? 0.5 : a, direct ? y : sg * sg);
    return direct ? sg * C * cf / v : 0.5 * exp(-a * log1p(-sg * sg)) - sg * C * cf;
}

__global__ void __launch_bounds__(H1_TC * H1_NC) h1_table_kernel(const double* __restrict__ dofs,
                                                                 double* __restrict__ tab, int emask)
{
    __shared__ double cosv[4 * H1_NC], f[H1_TC][H1_NC], cn[H1_TC][H1_NC];
    const int h = blockIdx.y >> 2, e = blockIdx.y & 3;
    if (!((emask >> e) & 1)) return;
    const double v = dofs[3 * h] + e;
    if (!(v <= H1_DOF_MAX + 4.0)) return;  // read by no record; also the normal limit
    const int lc = threadIdx.x / H1_NC, j = threadIdx.x % H1_NC;
    const int cell = blockIdx.x * H1_TC + lc;
    if (threadIdx.x < 4 * H1_NC) cosv[threadIdx.x] = cospi(threadIdx.x / (2.0 * H1_NC));
    __syncthreads();
    f[lc][j] = h1_value((cell + 0.5 + 0.5 * cosv[2 * j + 1]) * (1.0 / H1_CELLS), v, cf_t_const(v));
    __syncthreads();
    const double f0 = f[lc][H1_NC / 2];
    double s = 0.0;
    for (int i = 0; i < H1_NC; ++i) s += (f[lc][i] - f0) * cosv[(j * (2 * i + 1)) % (4 * H1_NC)];
    cn[lc][j] = s * (j ? 2.0 / H1_NC : 1.0 / H1_NC);
    __syncthreads();
    s = 0.0;
    for (int n = H1_NC - 1; n >= j; --n) s += cn[lc][n] * h1_cheb[n][j];
    s *= (double)(1 << j);  // x = 2 t
    tab[(size_t)blockIdx.y * H1_SIZE + cell * H1_NC + j] = j ? s : s + f0;
}

// The FP32 tables (internal.cuh, H32_*): cubics through H at the 4 Chebyshev nodes of each cell.
// Blocks of 32 cells (blockIdx.x), a thread per node.  Table blockIdx.y: 4h + e at dof
// nu_h + p + e where emask has bit e (emask > 0), else case blockIdx.y at dofs[blockIdx.y] + 1.
__global__ void __launch_bounds__(128) h32_table_kernel(const double* __restrict__ dofs, float4* __restrict__ tab,
                                                        float* __restrict__ scale, int emask)
{
    __shared__ double f[32][4];
    const int e = blockIdx.y & 3;
    if (emask && !((emask >> e) & 1)) return;
    const double v = emask ? dofs[3 * (blockIdx.y >> 2)] + e : dofs[blockIdx.y] + 1.0;
    if (!(v < INFINITY)) return;  // the normal limit reads no table
    const int lc = threadIdx.x >> 2, j = threadIdx.x & 3;
    const int cell = blockIdx.x * 32 + lc;
    const double h = h32_sigma_max(v) / H32_CELLS;
    const double x4[2] = {0.9238795325112867, 0.3826834323650898};  // cos(pi/8), cos(3 pi/8)
    const double x = j == 0 ? x4[0] : j == 1 ? x4[1] : j == 2 ? -x4[1] : -x4[0];
    f[lc][j] = h1_value((cell + 0.5 + 0.5 * x) * h, v, cf_t_const(v));
    __syncthreads();
    if (threadIdx.x < 32) {
        const double* g = f[threadIdx.x];
        // even and odd parts in x = 2 t at x4[0], x4[1]: a + b x^2 and x (c + d x^2)
        const double e0 = 0.5 * (g[0] + g[3]), e1 = 0.5 * (g[1] + g[2]);
        const double o0 = 0.5 * (g[0] - g[3]) / x4[0], o1 = 0.5 * (g[1] - g[2]) / x4[1];
        const double q0 = x4[0] * x4[0], q1 = x4[1] * x4[1];
        const double b = (e0 - e1) / (q0 - q1), d = (o0 - o1) / (q0 - q1);
        tab[(size_t)blockIdx.y * H32_CELLS + blockIdx.x * 32 + threadIdx.x] =
            make_float4((float)(e1 - b * q1), (float)(2.0 * (o1 - d * q1)), (float)(4.0 * b), (float)(8.0 * d));
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) scale[blockIdx.y] = (float)(1.0 / h);
}
