// estep_t2.cu -- T_2 records: a warp per record (quadrature nodes over lanes), or in FP32
// the records' quadrature pieces dealt to groups of lanes.
#include "internal.cuh"
#include "special.cuh"

template <typename R>
__global__ void __launch_bounds__(256) t2_records_kernel(RecSet r, IntegArgs a)
{
    const int lane = threadIdx.x & (CF_WARP - 1);
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const bool f32 = sizeof(R) == sizeof(float);
    const R* glx = f32 ? (const R*)a.glx32 : (const R*)a.glx64;
    const R* glw = f32 ? (const R*)a.glw32 : (const R*)a.glw64;
    const R* cst = f32 ? (const R*)a.cst32 : (const R*)a.cst64;
    unsigned long long nodes = 0;  // this warp's quadrature nodes (profiler count)
    for (long long i = warp; i < r.nrec; i += nwarps) {
        const R* c = cst + r.tab[i] * CST_STRIDE;
        R h, k, rho, nu, omr2, cr;
        if (f32 && r.t2f) {
            // FP32 record fields written by the plan: no FP64 instruction here
            const float4 u0 = r.t2f[2 * i], u1 = r.t2f[2 * i + 1];
            h = u0.x; k = u0.y; rho = u0.z; nu = u0.w; omr2 = u1.x; cr = u1.y;
        } else {
            const double h64 = r.bt[2 * i], k64 = r.bt[2 * i + 1];
            const double rho64 = a.F[r.fac[i] + 2];  // L[1][0] of the 2 x 2 correlation factor
            h = (R)h64; k = (R)k64; rho = (R)rho64; nu = (R)r.dof[i];
            omr2 = (R)((1.0 - rho64) * (1.0 + rho64));
            cr = (R)(h64 * (rho64 > 0.0 ? rho64 : -rho64) - (rho64 > 0.0 ? k64 : -k64));
        }
        const int ti = a.h32_case ? r.tab[i] : r.tab[i] / 3 * 4 + r.tab[i] % 3 + 1;
        const float4* tab = f32 && a.h32tab ? a.h32tab + (size_t)ti * H32_CELLS : nullptr;
        int nn = 2 * a.t2n;
        const double v = isinf(nu) ? phi2_warp<R>(h, k, rho, a.t2n, glx, glw, lane)
                                   : t2cdf_warp<R>(h, k, rho, nu, omr2, cr, c[CST_LGB], c[CST_LGB1], c[CST_C2], a.t2n,
                                       glx, glw, f32 ? T2_NH : a.t2n,
                                       f32 ? (const R*)a.glx32h : glx, f32 ? (const R*)a.glw32h : glw,
                                       lane, tab, tab ? a.h32scale[ti] : 0.0f, &nn, f32 ? a.t2n_lo : 0, f32 ? (const R*)a.glx32l : nullptr,
                                       f32 ? (const R*)a.glw32l : nullptr);
        nodes += (unsigned long long)nn;
        if (lane == 0) {
            if (r.res32) r.res32[i] = (float)v;
            else r.res[i] = v;
            if (r.se) r.se[i] = 0.0;
        }
    }
    if (a.nodes && lane == 0 && nodes) atomicAdd(a.nodes, nodes);
}

// FP32 T_2 records (finite dof), scheduled by quadrature piece.  A warp takes a chunk of
// up to 128 records; lane l sets up records l, l + 32, ... (the angles of the split, the pieces'
// lengths and node counts, once per record), the chunk's pieces (one or two per record,
// 8 to 64 nodes each) are ordered by node set and dealt to the warp's 32/L groups of L
// lanes, a group sums its piece's nodes (lane sub takes nodes sub, sub + L, ...), and the
// record's value is C_nu (piece 0 + piece 1).  Dealing pieces rather than records keeps
// the groups of a round on equal node counts: a record with one piece no longer idles its
// lanes while a neighbour's second piece runs.  The same L gives the same bits.
namespace {
constexpr int T2P_WARPS = 8;
constexpr int T2P_R = 4;                 // records per lane of a warp's chunk
constexpr int T2P_CH = T2P_R * CF_WARP;  // records per warp chunk
// a record's set-up fields, one array per field (consecutive records in distinct banks)
enum { T2F_ANC, T2F_L0, T2F_L1, T2F_D0, T2F_SC, T2F_NU, T2F_LGB1, T2F_N };
constexpr int T2P_NMAX = 64;  // nodes per piece at most (t2_nodes <= 64, T2_NH = 64)
// node sets: the classes 0-4 of t2_lo_class, then t2n nodes, then the graded pieces' T2_NH
constexpr int T2P_NK = T2_LO_NCLS + 2, T2P_KN = T2_LO_NCLS, T2P_KG = T2_LO_NCLS + 1;
}  // namespace

// TAB: the inner T_1 from the per-dof tables of H (a.h32tab), else by its continued fraction.
// With c = zs^2/(nu + 1), r = 1/sqrt(1 + c sin^2(phi - phi*)) and sigma = sqrt(c)
// |sin(phi - phi*)| r the node's T_1(-|z|) is T = r^(nu+1) H(sigma), and z's sign is one per
// piece: the integrand is sin^(nu-1)(phi) (0 + T) or (1 - T).  A lane takes two neighbouring
// nodes at a time in packed FP32.  The kernel was bound by instruction issue: 77 instructions a
// node (two folded sines, two lg2, two ex2, a Hermite interpolation) are about 40, and a record's set-up
// takes two arctangents (cf_atan2_f32) instead of three from the library.  The set-up keeps full
// FP32 precision (Newton steps, sqrtf, remainders; 2.19 -> 2.22 ms): u = alpha / alpha_s is as exact as
// its two records.
// p = 16, q = 2, g = 8, n = 2,000,000 (3.2e7 records, 25 nodes each) on a GB300: 2.66 -> 2.1 ms
// (2.2 at the parameters of the comparison above);
// a node is 60 cycles of a scheduler (FMA about 40, MUFU 32), a record's set-up, ordering and
// rounds about 15 nodes' worth.
template <int L, bool TAB>
__global__ void __launch_bounds__(T2P_WARPS * CF_WARP, 4) t2_pieces_kernel(RecSet r, IntegArgs a, int rows)
{
    constexpr int G = CF_WARP / L;
    __shared__ float srf[T2P_WARPS][T2F_N][T2P_CH];
    __shared__ int srt[T2P_WARPS][T2P_CH];                     // 2 table index + sign bit
    __shared__ unsigned char srk[T2P_WARPS][2 * T2P_CH];       // node set of piece (record << 1) | pc
    __shared__ __align__(8) float sgx[T2P_NK][T2P_NMAX], sgw[T2P_NK][T2P_NMAX];  // the node sets
    __shared__ float spsum[T2P_WARPS][T2P_CH][2];
    __shared__ unsigned char sitem[T2P_WARPS][2 * T2P_CH];  // (record << 1) | piece
    const int lane = threadIdx.x & (CF_WARP - 1), wib = threadIdx.x >> 5;
    const int sub = lane & (L - 1), grp = lane / L;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    float (*Rf)[T2P_CH] = srf[wib];
    int* Rt = srt[wib];
    unsigned char* Rk = srk[wib];
    float (*P)[2] = spsum[wib];
    unsigned char* items = sitem[wib];
    auto count = [&](int kd) { return kd < T2P_KN ? t2_lo_nodes(kd) : kd == T2P_KN ? a.t2n : T2_NH; };
    for (int e = threadIdx.x; e < T2P_NK * T2P_NMAX; e += blockDim.x) {
        const int kd = e / T2P_NMAX, i = e % T2P_NMAX;
        float x = 0.0f, w = 0.0f;
        if (kd < T2P_KN) {
            if (a.t2n_lo > 0 && i < t2_lo_nodes(kd)) { x = a.glx32l[t2_lo_off(kd) + i]; w = a.glw32l[t2_lo_off(kd) + i]; }
        } else if (kd == T2P_KN) {
            if (i < a.t2n) { x = a.glx32[i]; w = a.glw32[i]; }
        } else if (i < T2_NH) {
            const float u = a.glx32h[i];
            x = u * u * u; w = a.glw32h[i] * (3.0f * u * u);
        }
        sgx[kd][i] = x;
        sgw[kd][i] = w;
    }
    __syncthreads();
    unsigned long long nodes = 0;  // this lane's records' quadrature nodes (profiler count)
    const int chunk = rows * CF_WARP;  // records of a warp's chunk, at most T2P_CH
    for (long long base = warp * chunk; base < r.nrec; base += nwarps * chunk) {
        // phase 1: set-up of records lane, lane + 32, ...
        int np[T2P_R], kind[T2P_R][2];
        float C2[T2P_R], lim[T2P_R];
        bool limit[T2P_R];
#pragma unroll
        for (int m = 0; m < T2P_R; ++m) {
            const int rr = lane + m * CF_WARP;
            const long long i = base + rr;
            np[m] = 0; kind[m][0] = kind[m][1] = T2P_KN; C2[m] = 0.0f; lim[m] = 0.0f; limit[m] = false;
            if (m >= rows || i >= r.nrec) continue;
            const float* c = a.cst32 + r.tab[i] * CST_STRIDE;
            float h, k, rho, nu, omr2, cr;
            if (r.t2f) {  // FP32 record fields written by the plan
                const float4 u0 = r.t2f[2 * i], u1 = r.t2f[2 * i + 1];
                h = u0.x; k = u0.y; rho = u0.z; nu = u0.w; omr2 = u1.x; cr = u1.y;
            } else {
                const double h64 = r.bt[2 * i], k64 = r.bt[2 * i + 1];
                const double rho64 = a.F[r.fac[i] + 2];  // L[1][0] of the 2 x 2 correlation factor
                h = (float)h64; k = (float)k64; rho = (float)rho64; nu = (float)r.dof[i];
                omr2 = (float)((1.0 - rho64) * (1.0 + rho64));
                cr = (float)(h64 * (rho64 > 0.0 ? rho64 : -rho64) - (rho64 > 0.0 ? k64 : -k64));
            }
            C2[m] = c[CST_C2];
            if (rho >= 1.0f || rho <= -1.0f) {  // the |rho| = 1 limits: no pieces
                limit[m] = true;
                if (rho >= 1.0f) {
                    lim[m] = t1cdf_dev<float>(h < k ? h : k, nu, c[CST_LGB]);
                } else {
                    const float v = t1cdf_dev<float>(h, nu, c[CST_LGB]) + t1cdf_dev<float>(k, nu, c[CST_LGB]) - 1.0f;
                    lim[m] = v > 0.0f ? v : 0.0f;
                }
                continue;
            }
            const bool graded = fabsf(rho) > 0.99f;
            // fewer nodes where the integrand is smooth enough (t2_lo_class, per piece)
            const bool lo = a.t2n_lo > 0 && !graded && fabsf(rho) < T2_LO_RHO && nu >= T2_LO_DOF_MIN &&
                            nu <= T2_LO_DOF_MAX;
            // the angles of t2_setup: D = phi_h - phi*, and phi* or phi_h as the pieces' anchor
            const float sg = rho > 0.0f ? 1.0f : -1.0f, ar = fabsf(rho), sn = sqrt_newton(nu);
            const float D = cf_atan2_f32(sn * cr, fmaf(sg * h, k, ar * nu));
            const bool split = rho != 0.0f && D > 0.0f;
            const float anc = cf_atan2_f32(split ? ar * sn : sn, split ? -sg * k : -h);
            const float c1 = fmaf(rho * rho, nu, k * k) * rcp_newton(omr2 * nu);  // zs^2 / (nu + 1)
            np[m] = split ? 2 : 1;
            kind[m][0] = graded ? T2P_KG : lo ? t2_lo_class(anc, nu, c1 * (nu + 1.0f)) : T2P_KN;
            kind[m][1] = graded ? T2P_KG : lo ? t2_lo_class(D, nu, c1 * (nu + 1.0f)) : T2P_KN;
            nodes += (unsigned long long)(count(kind[m][0]) + (split ? count(kind[m][1]) : 0));
            Rf[T2F_ANC][rr] = anc;
            Rf[T2F_L0][rr] = -anc; Rf[T2F_L1][rr] = D;
            Rf[T2F_D0][rr] = split ? 0.0f : D;
            Rf[T2F_SC][rr] = sqrtf(c1);
            Rf[T2F_NU][rr] = nu; Rf[T2F_LGB1][rr] = c[CST_LGB1];
            // z > 0 on the first piece: bit 0 (the second piece's sign is the opposite)
            const bool pos0 = rho == 0.0f ? k > 0.0f : sg > 0.0f;
            const int ti = a.h32_case ? r.tab[i] : r.tab[i] / 3 * 4 + r.tab[i] % 3 + 1;
            Rt[rr] = 2 * ti + (pos0 ? 1 : 0);
            Rk[2 * rr] = (unsigned char)kind[m][0];
            Rk[2 * rr + 1] = (unsigned char)kind[m][1];
        }
        // the chunk's pieces, grouped by node set: a counting sort with the seven sets' counts (at most
        // 256 each) in 9-bit fields of one 64-bit word, scanned over the lanes once for all sets
        unsigned long long mine = 0;
#pragma unroll
        for (int m = 0; m < T2P_R; ++m)
#pragma unroll
            for (int pc = 0; pc < 2; ++pc)
                if (pc < np[m]) mine += 1ull << (9 * kind[m][pc]);
        unsigned long long incl = mine;
#pragma unroll
        for (int o = 1; o < CF_WARP; o <<= 1) {
            const unsigned long long v = __shfl_up_sync(CF_FULL, incl, o);
            if (lane >= o) incl += v;
        }
        const unsigned long long total = __shfl_sync(CF_FULL, incl, CF_WARP - 1);
        // field k of this product is the number of pieces in sets 0..k
        const unsigned long long upto = total * 0x0040201008040201ull;
        const int M = (int)(upto >> 54) & 511;  // field 6: the last set
        unsigned long long pos = (upto << 9) + incl - mine;  // field k: this lane's next place in set k
#pragma unroll
        for (int m = 0; m < T2P_R; ++m)
#pragma unroll
            for (int pc = 0; pc < 2; ++pc)
                if (pc < np[m]) {
                    items[(pos >> (9 * kind[m][pc])) & 511] = (unsigned char)(((lane + m * CF_WARP) << 1) | pc);
                    pos += 1ull << (9 * kind[m][pc]);
                }
        __syncwarp();
        // phase 2: rounds of G pieces, one per group
        for (int it0 = 0; it0 < M; it0 += G) {
            const int it = it0 + grp;
            float acc = 0.0f;
            int rr = 0, pc = 0;
            if (it < M) {
                rr = items[it] >> 1;
                pc = items[it] & 1;
                const int kd = Rk[items[it]];
                const int nn = count(kd);
                const float* gx = sgx[kd];
                const float* gw = sgw[kd];
                const float anc = Rf[T2F_ANC][rr];
                const float Lp = pc ? Rf[T2F_L1][rr] : Rf[T2F_L0][rr];
                const float d0 = pc ? 0.0f : Rf[T2F_D0][rr];
                const float sc = Rf[T2F_SC][rr], nu = Rf[T2F_NU][rr];
                const float num1 = nu - 1.0f, nu1 = nu + 1.0f;
                const bool pos = ((Rt[rr] ^ pc) & 1) != 0;
                // the nodes' sum is scaled by |L| once, below; graded sets are stored as u^3, 3 u^2 w
                if constexpr (TAB) {
                    const int ti = Rt[rr] >> 1;
                    const float4* __restrict__ tab = a.h32tab + (size_t)ti * H32_CELLS;
                    const float scale = __ldg(a.h32scale + ti);
                    const float A = pos ? 1.0f : 0.0f, B = pos ? -1.0f : 1.0f;
                    f32x2 acc2 = 0ull;
                    for (int t = 2 * sub; t < nn; t += 2 * L) {  // an odd count is padded with weight 0
                        const f32x2 off = mul2(*reinterpret_cast<const f32x2*>(gx + t), pk2(Lp));
                        const f32x2 sp = sin2_signed(add2(off, pk2(anc)));
                        const f32x2 q = mul2(sin2_signed(add2(off, pk2(d0))), pk2(sc));
                        float D0, D1, s0, s1;
                        up2(fma2(q, q, pk2(1.0f)), D0, D1);
                        up2(mul2(sp, sp), s0, s1);
                        const float r0 = rsqrt_approx(D0), r1 = rsqrt_approx(D1);
                        const f32x2 rr2 = pk2(r0, r1);
                        float e0, e1, g0, g1, u0, u1;
                        // the powers through the logarithms of the squares: lg2's absolute error near 1
                        // enters with (nu - 1)/2
                        up2(mul2(pk2(ptx_lg2_approx(s0), ptx_lg2_approx(s1)), pk2(0.5f * num1)), e0, e1);
                        up2(mul2(pk2(ptx_lg2_approx(D0), ptx_lg2_approx(D1)), pk2(-0.5f * num1)), g0, g1);
                        // H(sigma) as h32_eval
                        up2(fma2(mul2(q & 0x7fffffff7fffffffull, rr2), pk2(scale), pk2(-0.5f)), u0, u1);
                        const f32x2 u = pk2(fminf(u0, H32_U_MAX), fminf(u1, H32_U_MAX));
                        const f32x2 mm = add2(u, pk2(12582912.0f));
                        float m0, m1, t0, t1;
                        up2(mm, m0, m1);
                        up2(fma2(add2(mm, pk2(-12582912.0f)), pk2(-1.0f), u), t0, t1);
                        const float4 c0 = __ldg(tab + (__float_as_int(m0) & (H32_CELLS - 1)));
                        const float4 c1 = __ldg(tab + (__float_as_int(m1) & (H32_CELLS - 1)));
                        const f32x2 H = pk2(fmaf(fmaf(fmaf(c0.w, t0, c0.z), t0, c0.y), t0, c0.x),
                                            fmaf(fmaf(fmaf(c1.w, t1, c1.z), t1, c1.y), t1, c1.x));
                        const f32x2 T = mul2(mul2(pk2(ptx_ex2_approx(g0), ptx_ex2_approx(g1)), mul2(rr2, rr2)), H);
                        const f32x2 f = mul2(pk2(ptx_ex2_approx(e0), ptx_ex2_approx(e1)), fma2(T, pk2(B), pk2(A)));
                        acc2 = fma2(*reinterpret_cast<const f32x2*>(gw + t), f, acc2);
                    }
                    float a0, a1;
                    up2(acc2, a0, a1);
                    acc = a0 + a1;
                } else {
                    const float lgb1 = Rf[T2F_LGB1][rr], zs = sc * sqrtf(nu1);
                    for (int t = sub; t < nn; t += L) {
                        const float off = Lp * gx[t];
                        const float sp = cf_sin_pi(anc + off), sd = cf_sin_pi(d0 + off);
                        const float t1 = t1cdf_dev<float>(pos ? fabsf(zs * sd) : -fabsf(zs * sd), nu1, lgb1);
                        acc = fmaf(gw[t], ptx_ex2_approx(num1 * ptx_lg2_approx(sp)) * t1, acc);
                    }
                }
                acc *= fabsf(Lp);
            }
            acc = group_sum<L>(acc);
            if (it < M && sub == 0) P[rr][pc] = acc;
        }
        __syncwarp();
        // phase 3: records lane, lane + 32, ...
#pragma unroll
        for (int m = 0; m < T2P_R; ++m) {
            const int rr = lane + m * CF_WARP;
            const long long i = base + rr;
            if (m >= rows || i >= r.nrec) continue;
            float v;
            if (limit[m]) v = lim[m];
            else v = C2[m] * (np[m] == 2 ? P[rr][0] + P[rr][1] : P[rr][0]);
            if (r.res32) r.res32[i] = v;
            else r.res[i] = (double)v;
            if (r.se) r.se[i] = 0.0;
        }
        __syncwarp();
    }
    if (a.nodes) {
#pragma unroll
        for (int o = CF_WARP / 2; o > 0; o >>= 1) nodes += __shfl_xor_sync(CF_FULL, nodes, o);
        if (lane == 0 && nodes) atomicAdd(a.nodes, nodes);
    }
}

// FP64 T_2 records of a finite dof (the pieces of t2_setup, the same nodes).  With v = nu + 1
// and c = zs^2/v, the inner T_1 of a node is, where its argument z = zs sin(phi - phi*) is
// negative, sin^v(phi_z) H(sigma) with sin phi_z = r = 1/sqrt(1 + c sin^2(phi - phi*)) and
// sigma = sqrt(c) |sin(phi - phi*)| r, so the node's integrand is
//   sin^(nu-1)(phi) T_1 = (sin(phi) r)^(nu-1) r^2 H(sigma):
// one logarithm, one exponential, one rsqrt and a table polynomial.  On a piece where z > 0
// it is sin^(nu-1)(phi) (1 - T_1(-z)): the same integrand subtracted from the piece's part of
// the univariate T_1(.; nu), also by H.  z changes sign at phi* only, so its sign is one per
// piece; 1 - T_1(-z) >= 1/2 there, so the subtraction costs at most one bit.  Where the piece's
// part is itself a difference T_1(h) - T_1(k / rho) that loses more than two bits (rho < 0, phi*
// near phi_h), the factor 1 - T_1(-z) is formed at the nodes, a second logarithm and exponential.
//
// Bound by the FP64 pipe (1/64 of the FP32 rate): a node was a continued fraction with six
// divisions an iteration, about 1460 FP64 slots, and is about 80.  A warp takes up to 32
// records: lane l sets up record l (two arctangents, three square roots, the univariate
// part), then the warp runs each record's nodes over its lanes.  Measured on a GB300:
// p = 16, q = 2, g = 8, n = 20,000 (3.2e5 records): 72.1 ms with the continued fraction and 97
// nodes a record, 7.5 through H with log() and exp(), 3.8 with node_log, node_exp and 57 nodes
// (t2_lo_f64); p = q = g = 2, n = 1000 (4000 records): 1.48 -> 0.12 ms.
constexpr int T2D_WARPS = 8;
enum { T2D_ANC0, T2D_PHIS, T2D_L0, T2D_L1, T2D_D0, T2D_SC, T2D_NU, T2D_N };

// The t2n = 64 nodes of a piece are 32 (one round of the warp instead of two) where the
// Gauss-Legendre error of 32 stays below 1e-16 of the record's T_2: 10 <= dof <= 64,
// |rho| < 0.9 and L^2 (dof - 1 + 0.5 zs^2) <= 90.  Measured in 80-bit arithmetic on 24,000 records of the
// two distributions of fit_t2_classes.py: below 1e-16 up to a root of 10.2 (kept: 9.5),
// 67 % of the pieces there.  Only without a node count in the options (a.t2n_lo).
constexpr int T2D_NLO = 32;
__device__ __forceinline__ bool t2_lo_f64(double L, double nu, double zs2) { return L * L * (nu - 1.0 + 0.5 * zs2) <= 90.0; }

// records outside the tables (|rho| = 1, dof above H1_DOF_MAX or infinite): the general routines
static __device__ __noinline__ double t2_general_f64(const RecSet& r, const IntegArgs& a, long long i, int lane, int* nn)
{
    const double* c = a.cst64 + r.tab[i] * CST_STRIDE;
    const double h = r.bt[2 * i], k = r.bt[2 * i + 1], rho = a.F[r.fac[i] + 2];
    if (isinf(r.dof[i])) {
        *nn = 2 * a.t2n;
        return phi2_warp<double>(h, k, rho, a.t2n, a.glx64, a.glw64, lane);
    }
    return t2cdf_warp<double>(h, k, rho, r.dof[i], (1.0 - rho) * (1.0 + rho),
                              h * (rho > 0.0 ? rho : -rho) - (rho > 0.0 ? k : -k), c[CST_LGB], c[CST_LGB1], c[CST_C2],
                              a.t2n, a.glx64, a.glw64, a.t2n, a.glx64, a.glw64, lane, nullptr, 0.0f, nn);
}

// chunk: records per warp, 1..32
__global__ void __launch_bounds__(T2D_WARPS * CF_WARP, 2) t2_records_h1_kernel(RecSet r, IntegArgs a, int chunk)
{
    __shared__ NodeTables nt;
    __shared__ double sf[T2D_WARPS][T2D_N][CF_WARP];
    const int lane = threadIdx.x & (CF_WARP - 1), wib = threadIdx.x >> 5;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    double (*R)[CF_WARP] = sf[wib];
    node_tables_init(nt);
    unsigned long long nodes = 0;  // this warp's quadrature nodes (profiler count)
    for (long long base = warp * chunk; base < r.nrec; base += nwarps * chunk) {
        const int cnt = r.nrec - base < chunk ? (int)(r.nrec - base) : chunk;
        // bits: 0 split, 1 the first piece's z > 0 (the second one's is the opposite), 2 graded,
        // 3 general routine, 4 the second piece's factor 1 - T_1(-z) at the nodes, 5 and 6 the first
        // and second piece with T2D_NLO nodes
        int kind = 0, tab = 0;
        double C2 = 0.0, part = 0.0;
        if (lane < cnt) {
            const long long i = base + lane;
            const double h = r.bt[2 * i], k = r.bt[2 * i + 1], nu = r.dof[i];
            const double rho = a.F[r.fac[i] + 2];  // L[1][0] of the 2 x 2 correlation factor
            tab = r.tab[i];
            C2 = a.cst64[tab * CST_STRIDE + CST_C2];
            tab = tab / 3 * 4 + tab % 3;  // the table at this dof; the next one at dof + 1
            if (!(fabs(rho) < 1.0) || !(nu <= H1_DOF_MAX)) {
                kind = 8;
            } else {
                const double omr2 = (1.0 - rho) * (1.0 + rho), ar = fabs(rho), sg = rho > 0.0 ? 1.0 : -1.0;
                const double cr = h * ar - sg * k, sn = sqrt(nu);
                // D = phi_h - phi*, as in t2_setup; then the one angle that the pieces need
                const double D = atan2(sn * cr, sg * h * k + ar * nu);
                const bool split = rho != 0.0 && D > 0.0;
                const double anc = split ? atan2(ar * sn, -sg * k) : atan2(sn, -h);
                const double R2 = rho * rho * nu + k * k;
                const bool pos0 = rho == 0.0 ? k > 0.0 : sg > 0.0;
                kind = (split ? 1 : 0) | (pos0 ? 2 : 0) | (ar > 0.99 ? 4 : 0);
                R[T2D_ANC0][lane] = anc;
                R[T2D_PHIS][lane] = anc;
                R[T2D_L0][lane] = -anc;
                R[T2D_L1][lane] = D;
                R[T2D_D0][lane] = split ? 0.0 : D;
                const double c1 = R2 / (omr2 * nu);  // zs^2 / (nu + 1)
                R[T2D_SC][lane] = sqrt(c1);
                if (a.t2n_lo && nu >= 10.0 && nu <= 64.0 && ar < 0.9)
                    kind |= (t2_lo_f64(anc, nu, c1 * (nu + 1.0)) ? 32 : 0) | (t2_lo_f64(D, nu, c1 * (nu + 1.0)) ? 64 : 0);
                R[T2D_NU][lane] = nu;
                if (pos0 || split) {  // a piece with z > 0: its part of T_1(.; nu)
                    const double* t1 = a.h1tab + (size_t)tab * H1_SIZE;
                    double th = 0.0, ts = 0.0;
                    const double rh = rsqrt(nu + h * h), rs = rsqrt(R2);
                    if (!split || !pos0) th = h1_tail(sn * rh, fabs(h) * rh, nu, t1);
                    if (split) ts = h1_tail(ar * sn * rs, fabs(k) * rs, nu, t1);
                    const bool xneg = -sg * k > 0.0;  // cos phi* > 0: x* = k / rho < 0
                    if (!split) part = h > 0.0 ? 1.0 - th : th;
                    else if (pos0) part = xneg ? ts : 1.0 - ts;
                    else {
                        part = h <= 0.0 ? th - ts : xneg ? (1.0 - th) - ts : ts - th;
                        if (part < 0.25 * (h <= 0.0 ? th : 1.0 - th)) {
                            part = 0.0;
                            kind |= 16;
                        }
                    }
                }
            }
        }
        __syncwarp();
        double mine = 0.0;  // lane l: the quadrature sum of record l
        for (int l = 0; l < cnt; ++l) {
            const int kd = __shfl_sync(CF_FULL, kind, l), tb = __shfl_sync(CF_FULL, tab, l);
            if (kd & 8) {
                int nn = 0;
                const double v = t2_general_f64(r, a, base + l, lane, &nn);
                nodes += (unsigned long long)nn;
                if (lane == l) mine = v;
                continue;
            }
            const double sc = R[T2D_SC][l], num1 = R[T2D_NU][l] - 1.0;
            const double* __restrict__ t2 = a.h1tab + (size_t)(tb + 1) * H1_SIZE;
            double acc = 0.0;
            for (int pc = 0; pc <= (kd & 1); ++pc) {
                const double anc = pc ? R[T2D_PHIS][l] : R[T2D_ANC0][l], d0 = pc ? 0.0 : R[T2D_D0][l];
                const double L = pc ? R[T2D_L1][l] : R[T2D_L0][l];
                double s = 0.0;
                const bool lo = (kd >> (5 + pc)) & 1;
                const int n = lo ? T2D_NLO : a.t2n;
                const double* __restrict__ gx = lo ? a.glx64l : a.glx64;
                const double* __restrict__ gw = lo ? a.glw64l : a.glw64;
                nodes += (unsigned long long)n;
                for (int t = lane; t < n; t += CF_WARP) {
                    const double u = gx[t];
                    double w = gw[t], um = u;
                    if (kd & 4) {  // nodes anchor + L u^3, weights 3 u^2
                        um = u * u * u;
                        w *= 3.0 * u * u;
                    }
                    const double off = L * um;
                    const double sp = cf_sin_pi(anc + off);  // both arguments lie in [-pi, pi]
                    const double q = sc * cf_sin_pi(d0 + off);
                    const double rr = rsqrt(fma(q, q, 1.0));
                    const double H = h1_eval(fabs(q) * rr, t2);
                    if (kd & pc << 4)
                        s = fma(w * node_exp<true>(num1 * node_log(fabs(sp), nt), nt), 1.0 - node_exp<true>(num1 * node_log(rr, nt), nt) * (rr * rr) * H, s);
                    else
                        s = fma(w * (rr * rr), node_exp<true>(num1 * node_log(fabs(sp) * rr, nt), nt) * H, s);
                }
                acc = fma(((kd >> 1) ^ pc) & !(kd & pc << 4) ? -fabs(L) : fabs(L), s, acc);
            }
            acc = warp_sum(acc);
            if (lane == l) mine = acc;
        }
        if (lane < cnt) {
            const long long i = base + lane;
            r.res[i] = kind & 8 ? mine : fma(C2, mine, part);
            if (r.se) r.se[i] = 0.0;
        }
        __syncwarp();
    }
    if (a.nodes && lane == 0 && nodes) atomicAdd(a.nodes, nodes);
}

// Lanes per FP32 T_2 piece (finite dof), a.t2_group in {2, 4, 8, 16}; 32 (or 0: the CFUSN
// model's records) = the warp-per-record kernel.
template <int L>
static void go_group(const RecSet& r, const IntegArgs& a, int nsm, cudaStream_t st)
{
    // records per lane of a chunk: as many as leave every SM its 32 resident warps (longer
    // chunks lose less in the rounds where node counts change and in the last one: p = 16, q = 2,
    // 6.4e6 records 0.472 ms at 2, 0.432 at 3, 0.424 at 4)
    const long long fill = 4LL * T2P_WARPS * nsm * CF_WARP;
    const int rows = (int)(r.nrec <= fill ? 1 : r.nrec >= T2P_R * fill ? T2P_R : (r.nrec + fill - 1) / fill);
    const long long per_block = (long long)T2P_WARPS * CF_WARP * rows;
    const long long need = (r.nrec + per_block - 1) / per_block, cap = 16LL * nsm;
    const int gb = (int)(need < cap ? need : cap);
    if (a.h32tab) t2_pieces_kernel<L, true><<<gb, T2P_WARPS * CF_WARP, 0, st>>>(r, a, rows);
    else t2_pieces_kernel<L, false><<<gb, T2P_WARPS * CF_WARP, 0, st>>>(r, a, rows);
}

cudaError_t launch_t2(const RecSet& r, const IntegArgs& a, int fp32, int blocks, int nsm, cudaStream_t st)
{
    if (!fp32 && a.h1tab) {
        // records per warp: a record's set-up takes a warp about as long as 8 records' nodes
        // over its lanes, so up to 32 share one; fewer where that would leave the SMs with
        // less than 4 warps each (one per scheduler keeps the FP64 pipes busy)
        long long ch = r.nrec / (4LL * nsm);
        ch = ch < 1 ? 1 : ch > CF_WARP ? CF_WARP : ch;
        const long long need = (r.nrec + ch * T2D_WARPS - 1) / (ch * T2D_WARPS);
        const long long cap = 8LL * nsm;
        t2_records_h1_kernel<<<(int)(need < cap ? need : cap), T2D_WARPS * CF_WARP, 0, st>>>(r, a, (int)ch);
        return cudaGetLastError();
    }
    const int L = a.t2_group;
    if (fp32 && L == 2) go_group<2>(r, a, nsm, st);
    else if (fp32 && L == 4) go_group<4>(r, a, nsm, st);
    else if (fp32 && L == 8) go_group<8>(r, a, nsm, st);
    else if (fp32 && L == 16) go_group<16>(r, a, nsm, st);
    else if (fp32) {
        t2_records_kernel<float><<<blocks, 256, 0, st>>>(r, a);
    } else {
        t2_records_kernel<double><<<blocks, 256, 0, st>>>(r, a);
    }
    return cudaGetLastError();
}
