// estep_fixup.cu -- FP64 re-evaluation of listed pairs.
//
// In FP32 mode the lattice products of a pair whose alpha_s (eq 4) is below
// 1e-35 leave the FP32 range; the combine kernel lists such pairs and this
// kernel recomputes every integral of those pairs in FP64, then the same
// assembly as the combine kernel.
//
// The list is usually short (none to a few dozen pairs of 1e5), and one pair is 8 million
// FP64 operations at q = 4 on a pipe of 2 lanes per SM and clock: a warp that did a whole
// pair held the E-step up for 6 to 38 ms while the rest of the GPU idled.  Up to fix_cap
// pairs are therefore cut into tasks, a warp each: an integral of dimension >= 3 into its
// shifts and those into parts of the points, a lower one whole.  The task sums go to
// a buffer; the warp that finishes a pair's last task adds them in their order (the
// same bits whichever warp it is) and assembles the pair.  Longer lists fill the GPU by
// themselves (FIX_CAP = 1024 pairs are 7 warps per SM): a warp takes a pair and runs its tasks
// in turn, with a buffer of its own.  Phi and its inverse come from tables (ncdf_tab): the FP64
// pipe is what a list of hundreds of pairs waits for.  Fix-up of one E-step on a GB300,
// parameters with strongly skewed components (a warp per pair -> tasks -> tasks and tables):
// p = q = g = 4, n = 200,000, single pass 12.2 -> 4.3 -> 3.4 ms; the same with recursion
// moments, n = 20,000, 26.9 -> 2.0 -> 1.7 ms; p = q = g = 6, n = 50,000, single pass
// 37.9 -> 18.4 -> 11.5 ms.
#include "estep_common.cuh"

// T_k(bt; 0, corr(Lc Lc^T), nu), k <= 2, in FP64, warp-cooperative
__device__ double tk_fp64(int k, const double* bt, const double* Lc, double nu, const EstepArgs& a, int lane)
{
    if (k == 0) return 1.0;
    if (k == 1) return isinf(nu) ? normcdf(bt[0]) : t1cdf_dev<double>(bt[0], nu, t1_lgb(nu));
    const double rho = Lc[2];
    if (isinf(nu)) return phi2_warp<double>(bt[0], bt[1], rho, a.t2n, a.glx64, a.glw64, lane);
    return t2cdf_warp<double>(bt[0], bt[1], rho, nu, (1.0 - rho) * (1.0 + rho),
                              bt[0] * (rho > 0.0 ? rho : -rho) - (rho > 0.0 ? bt[1] : -bt[1]), t1_lgb(nu),
                              t1_lgb(nu + 1.0), cf_t_const(nu), a.t2n, a.glx64, a.glw64, a.t2n, a.glx64, a.glw64, lane);
}

// Sums over the points i0 <= i < i1 of shift m of the lattice pass of T_K (the points and
// factors of tk_lattice_warp / tk_lattice_mom_warp): out[0] = sum f and, MOM, out[1] = sum f s^2,
// out[2] = sum f log s^2 (lrow given), out[3..] = sum f s rk y_r, then sum f rk^2 y_r y_c (c <= r).
// All lanes; lane 0 writes.
template <int K, bool MOM>
__device__ void lattice_part(const double* bt, const double* Lc, const EstepArgs& a, const double* crow,
                             const double* lrow, double rk, int m, int i0, int i1, int lane, double* out,
                             const NcdfTables& nq)
{
    constexpr int K2 = K * (K + 1) / 2, NY = MOM ? K : K - 1;
    double b[K], invd[K], Lf[K][K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
        b[r] = bt[r];
        invd[r] = 1.0 / Lc[r * K + r];
#pragma unroll
        for (int l = 0; l < K; ++l) Lf[r][l] = l < r ? Lc[r * K + l] : 0.0;
    }
    const int N = a.lat.N;
    const double invN = 1.0 / (double)N;
    double af = 0.0, aw = 0.0, al = 0.0, a1[K], a2[K2];
#pragma unroll
    for (int r = 0; r < K; ++r) a1[r] = 0.0;
#pragma unroll
    for (int r = 0; r < K2; ++r) a2[r] = 0.0;
    for (int i = i0 + lane; i < i1; i += CF_WARP) {
        const double s = crow[i];
        double y[K], f = 1.0;
#pragma unroll
        for (int r = 0; r < K; ++r) {
            double t = b[r] * s;
#pragma unroll
            for (int l = 0; l < r; ++l) t -= Lf[r][l] * y[l];
            const double e = ncdf_tab(t * invd[r], nq);
            f *= e;
            if (r < NY) {
                double x = (double)(((long long)i * a.lat.z[r + 1]) % N) * invN + a.shf64[m * CF_MAXDIM + r + 1];
                if (x >= 1.0) x -= 1.0;
                double v = (1.0 - fabs(2.0 * x - 1.0)) * e;
                v = v < Lim<double>::vmin() ? Lim<double>::vmin() : v;
                v = v > Lim<double>::one_minus_ulp() ? Lim<double>::one_minus_ulp() : v;
                y[r] = ncdfinv_tab(v, nq);
            }
            if (e <= Lim<double>::tiny()) f = 0.0;
        }
        af += f;
        if (MOM) {
            const double fs = f * s, w1 = fs * rk, w2 = f * (rk * rk);
            aw += fs * s;
            if (lrow) al += f * lrow[i];
#pragma unroll
            for (int r = 0; r < K; ++r) {
                a1[r] += w1 * y[r];
                const double t = w2 * y[r];
#pragma unroll
                for (int c = 0; c <= r; ++c) a2[r * (r + 1) / 2 + c] += t * y[c];
            }
        }
    }
    af = warp_sum(af);
    if (lane == 0) out[0] = af;
    if (MOM) {
        aw = warp_sum(aw);
        al = warp_sum(al);
        if (lane == 0) { out[1] = aw; out[2] = al; }
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const double v = warp_sum(a1[r]);
            if (lane == 0) out[3 + r] = v;
        }
#pragma unroll
        for (int r = 0; r < K2; ++r) {
            const double v = warp_sum(a2[r]);
            if (lane == 0) out[3 + K + r] = v;
        }
    }
}

template <bool MOM>
__device__ void lattice_part_k(int k, const double* bt, const double* Lc, const EstepArgs& a, const double* crow,
                               const double* lrow, double rk, int m, int i0, int i1, int lane, double* out,
                               const NcdfTables& nq)
{
    switch (k) {
    case 3: lattice_part<3, MOM>(bt, Lc, a, crow, lrow, rk, m, i0, i1, lane, out, nq); break;
    case 4: lattice_part<4, MOM>(bt, Lc, a, crow, lrow, rk, m, i0, i1, lane, out, nq); break;
    case 5: lattice_part<5, MOM>(bt, Lc, a, crow, lrow, rk, m, i0, i1, lane, out, nq); break;
    case 6: lattice_part<6, MOM>(bt, Lc, a, crow, lrow, rk, m, i0, i1, lane, out, nq); break;
    case 7: lattice_part<7, MOM>(bt, Lc, a, crow, lrow, rk, m, i0, i1, lane, out, nq); break;
    default: lattice_part<8, MOM>(bt, Lc, a, crow, lrow, rk, m, i0, i1, lane, out, nq); break;
    }
}

// A pair's integral: dimension, dof, chi table (0..2 from the component's first), factor
// offset and standardised limits.  Numbered as its tasks run: alpha_s, alpha, then level 1 (r), then
// level 2 (r, s); density passes and the single pass have alpha_s's only.
__device__ void fix_integral(const EstepArgs& a, const double* F, const double* c, double d, int n, int& k,
                             double& dof, int& tab, int& fac, double* bt)
{
    const int p = a.D.p, q = a.D.q, q1 = q - 1;
    const double nu1 = F[a.Ly.scal + SC_NU] + p;
    if (n < 2) {
        k = q; dof = nu1 + 2.0 * n; tab = 2 * n; fac = fac_l0(a.Ly);
        limits_l0(F, a.Ly, p, q, c, d, n, bt);
    } else if (n < 2 + q) {
        const int r = n - 2;
        k = q1; dof = nu1 + 1.0; tab = 1; fac = fac_l1(a.Ly, q, r);
        limits_l1(F, a.Ly, p, q, c, d, r, bt);
    } else {
        const int r = (n - 2 - q) / q1, s = (n - 2 - q) % q1;
        k = q - 2; dof = nu1; tab = 0; fac = fac_l2(a.Ly, q, r, s);
        limits_l2(F, a.Ly, p, q, c, d, r, s, bt);
    }
}

__device__ void fix_store(const EstepArgs& a, long long pid, const PairOut& o, double se)
{
    const int q = a.D.q;
    a.logf[pid] = o.logf;
    if (a.se) a.se[pid] = se;
    if (!(o.logf < INFINITY)) atomicOr(a.flags, KF_NAN);  // NaN or +inf; -inf is a null pair
    if (a.density_only) return;
    if (a.pr32) {
        store_pr32(a.pr32 + pid * pr32_width(q), q, o);
        return;
    }
    a.u[pid] = o.u;
    a.elogu[pid] = o.elogu;
    for (int k = 0; k < q; ++k) a.eu[pid * q + k] = o.eu[k];
    for (int k = 0; k < q * q; ++k) a.euu[pid * q * q + k] = o.euu[k];
}

// A listed pair's factors, squared distance, log t_p and limits' vector
struct FixPair {
    const double* F;
    int h;
    double c[CF_MAXQ], d, logtp;
};
__device__ void fix_pair(const EstepArgs& a, long long pid, FixPair& P)
{
    P.h = (int)(pid / a.D.n);
    P.F = a.F + (size_t)P.h * a.Ly.stride;
    pair_whiten(P.F, a.Ly, a.D.p, a.D.q, a.y + (size_t)(pid - (long long)P.h * a.D.n) * a.D.p, &P.d, P.c, &P.logtp);
}

// Task t of a pair: its sums to out.  LAT: with integrals of dimension >= 3.
template <bool LAT>
__device__ void fix_task(const EstepArgs& a, const FixArgs& x, const FixPair& P, int t, int lane, double* out,
                         const NcdfTables* nq)
{
    const int q = a.D.q;
    double bt[CF_MAXQ], dof;
    // the integral's number: 2 of dimension q, q of q - 1, the rest of q - 2
    int n = 0, k, tab, fac;
    for (;; ++n) {
        const int w = fix_tasks_k(n < 2 ? q : n < 2 + q ? q - 1 : q - 2, x);
        if (t < w) break;
        t -= w;
    }
    fix_integral(a, P.F, P.c, P.d, n, k, dof, tab, fac, bt);
    if (!LAT || k < 3) {
        const double v = tk_fp64(k, bt, P.F + fac, dof, a, lane);
        if (lane == 0) out[0] = v;
        return;
    }
    if constexpr (LAT) {
        const size_t NM = (size_t)a.lat.N * a.lat.M;
        const int m = t / x.parts, part = t % x.parts;
        const int i0 = (int)((long long)a.lat.N * part / x.parts), i1 = (int)((long long)a.lat.N * (part + 1) / x.parts);
        const double* crow = a.chi64 + (size_t)(3 * P.h + tab) * NM + (size_t)m * a.lat.N;
        if (a.single_pass && !a.density_only) {
            const double* lrow = a.lchi64 ? a.lchi64 + (size_t)(3 * P.h) * NM + (size_t)m * a.lat.N : nullptr;
            const double rk = isinf(dof) ? 1.0 : sqrt((dof + 2.0) / dof);
            lattice_part_k<true>(k, bt, P.F + fac, a, crow, lrow, rk, m, i0, i1, lane, out, *nq);
        } else {
            lattice_part_k<false>(k, bt, P.F + fac, a, crow, nullptr, 1.0, m, i0, i1, lane, out, *nq);
        }
    }
}

// T_k from its tasks' sums (nv doubles a task): the mean over the shifts and its standard error;
// all lanes
__device__ double fix_value(const EstepArgs& a, const FixArgs& x, int k, const double* part, double* se)
{
    if (se) *se = 0.0;
    if (k == 0) return 1.0;
    if (k < 3) return part[0];
    double mean = 0.0, m2 = 0.0;
    for (int m = 0; m < a.lat.M; ++m) {
        double s = 0.0;
        for (int u = 0; u < x.parts; ++u) s += part[(size_t)(m * x.parts + u) * x.nv];
        const double smean = s / (double)a.lat.N, delta = smean - mean;
        mean += delta / (double)(m + 1);
        m2 += delta * (smean - mean);
    }
    if (se) *se = a.lat.M > 1 ? sqrt(m2 / (double)(a.lat.M - 1) / (double)a.lat.M) : 0.0;
    return mean;
}

// The pair from its tasks' sums; all lanes, sm: CF_MAXQ + CF_MAXQ (CF_MAXQ + 1) / 2 + 3 doubles
__device__ void fix_assemble(const EstepArgs& a, const FixArgs& x, long long pid, const FixPair& P, const double* part,
                             int lane, double* sm)
{
    const int p = a.D.p, q = a.D.q, q1 = q - 1, h = P.h;
    const double *F = P.F, *c = P.c;
    const double d = P.d, logtp = P.logtp;
    double se = 0.0;
    const double alpha_s = fix_value(a, x, q, part, &se);
    PairOut o;
    if (a.single_pass && !a.density_only) {
        for (int v = lane; v < x.nv; v += CF_WARP) {  // sm[v]: sum v over the tasks, in order
            double s = 0.0;
            for (int t = 0; t < x.ntask; ++t) s += part[(size_t)t * x.nv + v];
            sm[v] = s;
        }
        __syncwarp();
        // m1 = L E[y/s], m2 = L E[y y^T/s^2] L^T (see tk_lattice_mom_warp)
        const double* Lc = F + fac_l0(a.Ly);
        const double* s1 = sm + 3;
        const double* s2 = sm + 3 + q;
        const double inv = sm[1] > 0.0 ? 1.0 / sm[1] : 0.0;
        double m[CF_MAXQ + CF_MAXQ * (CF_MAXQ + 1) / 2];
        for (int r = 0; r < q; ++r) {
            double v = 0.0;
            for (int l = 0; l <= r; ++l) v += Lc[r * q + l] * s1[l];
            m[r] = v * inv;
            for (int cc = 0; cc <= r; ++cc) {
                double w2 = 0.0;
                for (int i = 0; i <= r; ++i) {
                    double w = 0.0;
                    for (int l = 0; l <= cc; ++l) w += s2[i >= l ? i * (i + 1) / 2 + l : l * (l + 1) / 2 + i] * Lc[cc * q + l];
                    w2 += Lc[r * q + i] * w;
                }
                m[q + r * (r + 1) / 2 + cc] = w2 * inv;
            }
        }
        const double lw = a.lchi64 ? (sm[0] > 0.0 ? sm[2] / sm[0] : NAN) : NAN;
        pair_assemble_sp(F, a.Ly, p, q, c, d, logtp, alpha_s, sm[1] / ((double)a.lat.N * a.lat.M), m, o, lw);
        __syncwarp();
    } else {
        double alpha = 0.0, tq1[CF_MAXQ], tq2[CF_MAXQ * CF_MAXQ];
        if (!a.density_only) {
            const size_t wq = (size_t)fix_tasks_k(q, x) * x.nv, w1 = (size_t)fix_tasks_k(q1, x) * x.nv,
                         w2 = (size_t)fix_tasks_k(q - 2, x) * x.nv;
            alpha = fix_value(a, x, q, part + wq, nullptr);
            for (int r = 0; r < q && q1 > 0; ++r) {
                tq1[r] = fix_value(a, x, q1, part + 2 * wq + r * w1, nullptr);
                for (int s = 0; s < q1 && q > 2; ++s)
                    tq2[r * q1 + s] = fix_value(a, x, q - 2, part + 2 * wq + q * w1 + (size_t)(r * q1 + s) * w2, nullptr);
            }
        }
        pair_assemble(F, a.Ly, p, q, c, d, logtp, alpha_s, alpha, tq1, tq2, a.density_only,
                      a.cst64 + (size_t)(3 * h) * CST_STRIDE, o);
    }
    if (lane == 0) fix_store(a, pid, o, se);
}

// LAT: q >= 3.  At q <= 2 no integral needs the tables of Phi, which take about 50 us to build
// (longer than a short list), nor the lattice code's registers, and a pair's few values fit in
// shared memory, so that every warp of a long list has a pair.  One kernel for every q ->
// without them at q <= 2, normal limit (CFUSN) on a GB300: p = 16, q = 2, g = 4, n = 2000 (a few
// pairs listed) E-step 104 -> 56 us, density 88 -> 39; g = 8, n = 200,000 (long list) 46.8 -> 23.9 ms,
// 14.2 -> 8.1 (a warp per pair with all of a pair's integrals in one function: 86, 37 us; 28.3, 8.2 ms).
template <bool LAT>
__global__ void __launch_bounds__(128, LAT ? 2 : 4) fixup_kernel(EstepArgs a, FixArgs x, const int* count, const int* list)
{
    __shared__ double slot[4][CF_MAXQ + CF_MAXQ * (CF_MAXQ + 1) / 2 + 3 + CF_MAXSHIFT];
    static_assert(sizeof(slot) >= (NCDF_CELLS + 4) * H1_NC * sizeof(double), "scratch of ncdf_tables_init");
    const int cnt = *count;
    if (cnt == 0) return;
    const int lane = threadIdx.x & (CF_WARP - 1);
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    double* sm = slot[threadIdx.x >> 5];
    const NcdfTables* nq = nullptr;
    if constexpr (LAT) {
        __shared__ NcdfTables tables;
        ncdf_tables_init(tables, &slot[0][0]);
        nq = &tables;
    }
    FixPair P;
    if (cnt <= x.cap) {
        const long long total = (long long)cnt * x.ntask;
        for (long long t = warp; t < total; t += nwarps) {
            const int i = (int)(t / x.ntask), k = (int)(t % x.ntask);
            double* part = x.part + (size_t)i * x.ntask * x.nv;
            fix_pair(a, list[i], P);
            fix_task<LAT>(a, x, P, k, lane, part + (size_t)k * x.nv, nq);
            int last = 0;
            if (lane == 0) {
                __threadfence();
                last = atomicAdd(x.done + i, 1) == x.ntask - 1;
            }
            last = __shfl_sync(CF_FULL, last, 0);
            if (!last) continue;
            __threadfence();
            fix_assemble(a, x, list[i], P, part, lane, sm);
            if (lane == 0) x.done[i] = 0;  // ready for the next E-step
        }
        return;
    }
    // a warp per pair, its tasks in turn into a buffer of its own: shared memory at q <= 2 (2 + 2 q
    // values), else a pair's place in the sums' buffer
    const int use = !LAT || nwarps < x.cap ? nwarps : x.cap;
    if (warp >= use) return;
    double* part = LAT ? x.part + (size_t)warp * x.ntask * x.nv : sm;
    for (int i = warp; i < cnt; i += use) {
        fix_pair(a, list[i], P);
        for (int k = 0; k < x.ntask; ++k) fix_task<LAT>(a, x, P, k, lane, part + (size_t)k * x.nv, nq);
        __syncwarp();
        fix_assemble(a, x, list[i], P, part, lane, sm);
        __syncwarp();  // part is reused
    }
}

// density: the tasks of a density pass, else of a full E-step (single: single-pass moments)
FixArgs fix_args(int q, int single, int density, const Lattice& lat)
{
    FixArgs x{};
    x.parts = lat.M >= 64 ? 1 : 64 / lat.M;
    if (x.parts > (lat.N + 127) / 128) x.parts = (lat.N + 127) / 128;
    x.tasks = lat.M * x.parts;
    const bool mom = single && !density;
    x.nv = mom ? 3 + q + q * (q + 1) / 2 : 1;
    x.ntask = density || mom ? fix_tasks_k(q, x)
                             : 2 * fix_tasks_k(q, x) + q * fix_tasks_k(q - 1, x) + q * (q - 1) * fix_tasks_k(q - 2, x);
    return x;
}

cudaError_t launch_fixup(const EstepArgs& a, const FixArgs& x, const int* count, const int* list, int nsm,
                         cudaStream_t st, long long* launches)
{
    if (a.D.q >= 3) fixup_kernel<true><<<4 * nsm, 128, 0, st>>>(a, x, count, list);
    else fixup_kernel<false><<<4 * nsm, 128, 0, st>>>(a, x, count, list);
    ++*launches;
    return cudaGetLastError();
}
