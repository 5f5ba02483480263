// estep_mom32.cu -- lattice T_k with truncated moments (single-pass ratio
// estimators), k = 3..8, in float: a warp per two records, lattice points over lanes
// (see mom_pair_f32 in special.cuh).
#include "internal.cuh"
#include "special.cuh"

// Minimum resident blocks of 4 warps: the pass is bound by the FMA and MUFU pipes' latency as much
// as their rate, so resident warps count for more than registers (K = 6: 3 blocks of 164
// registers 102.7, 4 of 128 with spills 112.3, 5 of 96 108.4 Gpoints/s; K = 7: 2 blocks 73.5,
// 3 89.4, 4 89.1; K = 5: 3, 4, 5 blocks 130, 136, 142).  Rates on a GB300 (p = q, g = 4,
// 4 n >= 4e4 records) against a warp per record with scalar FP32, before: K = 3 .. 8
// 222, 167, 105, 85, 60, 50 -> 270, 200, 142, 112, 89, 71 Gpoints/s.
template <int K, int P>
__host__ __device__ constexpr int mom32_minb()
{
    return K == 3 ? (P == 1 ? 6 : 5) : K == 4 ? (P == 1 ? 6 : 4) : K == 5 ? 5 : K == 6 ? 4 : 3;
}

template <int K, bool SEL, bool LW, int P>
__global__ void __launch_bounds__(128, mom32_minb<K, P>()) lattice_mom_kernel_32(RecSet r, IntegArgs a)
{
    const int lane = threadIdx.x & (CF_WARP - 1);
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    __shared__ float slot[4][mom2_slot(K)];
    float* sm = slot[threadIdx.x >> 5];
    const long long nr = rec_count<SEL>(r);
    for (long long t = 2 * warp; t < nr; t += 2 * nwarps) {
        // two records of one component, else (the last one, a change of component) one by one
        const bool two = t + 1 < nr;
        const long long i0 = rec_index<SEL>(r, t), i1 = two ? rec_index<SEL>(r, t + 1) : i0;
        const bool pair = two && r.tab[i0] == r.tab[i1];
        for (int k = 0; k < (two && !pair ? 2 : 1); ++k)
            mom_pair_f32<K, K <= 4, P, LW>(r, a, k ? i1 : i0, pair || k ? i1 : i0, pair, lane, sm);
    }
}

// the selection-list instantiation only where a list is given
template <int K, int P>
static void go_p(const RecSet& r, const IntegArgs& a, int blocks, cudaStream_t st)
{
    // exact E[log W] (r.lw) only without a selection list (the surrogate excludes it)
    if (r.sel) lattice_mom_kernel_32<K, true, false, P><<<blocks, 128, 0, st>>>(r, a);
    else if (r.lw) lattice_mom_kernel_32<K, false, true, P><<<blocks, 128, 0, st>>>(r, a);
    else lattice_mom_kernel_32<K, false, false, P><<<blocks, 128, 0, st>>>(r, a);
}

// points in flight per lane: a.mom_p (1 or 2) with the coordinate table (K <= 4), else 1
template <int K>
static void go(const RecSet& r, const IntegArgs& a, int blocks, cudaStream_t st)
{
    if constexpr (K <= 4) {
        if (a.mom_p == 1) go_p<K, 1>(r, a, blocks, st);
        else go_p<K, 2>(r, a, blocks, st);
    } else {
        go_p<K, 1>(r, a, blocks, st);
    }
}

cudaError_t launch_mom32(int k, const RecSet& r, const IntegArgs& a, int blocks, cudaStream_t st)
{
    switch (k) {
    case 3: go<3>(r, a, blocks, st); break;
    case 4: go<4>(r, a, blocks, st); break;
    case 5: go<5>(r, a, blocks, st); break;
    case 6: go<6>(r, a, blocks, st); break;
    case 7: go<7>(r, a, blocks, st); break;
    case 8: go<8>(r, a, blocks, st); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}
