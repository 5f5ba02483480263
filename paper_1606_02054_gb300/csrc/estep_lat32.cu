// estep_lat32.cu -- lattice T_k records, k = 3..8, in float: a warp per two
// records, lattice points over lanes (see lattice_pair_f32 in special.cuh).  Bound by the MUFU
// pipe (per factor and record pair: 8 operations, 56 of its cycles) beside the FMA pipe (about
// 48).  Rates on a GB300 against a warp per record with scalar FP32, before: K = 3, 4, 5, 6, 8
// 261, 187, 140, 96, 58 -> 316, 226, 165, 134, 69 Gpoints/s.
#include "internal.cuh"
#include "special.cuh"

template <int K, bool SEL>
__global__ void __launch_bounds__(128) lattice_records_kernel_32(RecSet r, IntegArgs a)
{
    const int lane = threadIdx.x & (CF_WARP - 1);
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    __shared__ float slot[4][lat2_slot(K)];
    const long long nr = rec_count<SEL>(r);
    for (long long t = 2 * warp; t < nr; t += 2 * nwarps) {
        const bool two = t + 1 < nr;
        const long long i0 = rec_index<SEL>(r, t), i1 = two ? rec_index<SEL>(r, t + 1) : i0;
        float v[2], se[2];
        lattice_pair_f32<K>(r, a, i0, i1, lane, slot[threadIdx.x >> 5], v, se);
        if (lane < (two ? 2 : 1)) {
            const long long i = lane ? i1 : i0;
            r.res[i] = (double)(lane ? v[1] : v[0]);
            if (r.se) r.se[i] = (double)(lane ? se[1] : se[0]);
        }
    }
}

// the selection-list instantiation only where a list is given
template <int K>
static void go(const RecSet& r, const IntegArgs& a, int blocks, cudaStream_t st)
{
    if (r.sel) lattice_records_kernel_32<K, true><<<blocks, 128, 0, st>>>(r, a);
    else lattice_records_kernel_32<K, false><<<blocks, 128, 0, st>>>(r, a);
}

cudaError_t launch_lattice32(int k, const RecSet& r, const IntegArgs& a, int blocks, cudaStream_t st)
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
