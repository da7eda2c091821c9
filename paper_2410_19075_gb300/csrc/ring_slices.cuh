// Rings held by one thread-block cluster, every CTA a slice of consecutive nodes in
// its shared memory (RK4 in ring_cluster.cu, Dormand-Prince in ring_dp_cluster.cu):
// the slices' exact prefix offsets and the window sums across slices.
#pragma once
#include "ring_parts.cuh"

namespace simk {

constexpr int kClusterMaxCtas = 16;

// Exact offsets of the cluster's slices from their totals, by one warp: lane r
// holds the prefix in front of slice r as hi 2^sh + lo (ex_*), every lane the
// ring's total (tot_*).
template <int NQ> struct SliceOffsets {
    int64_t ex_hi[NQ], tot_hi[NQ];
    int ex_lo[NQ], tot_lo[NQ];
};
template <int NQ>
__device__ __forceinline__ void slice_offsets(const int64_t (*tot)[NQ], int CL, int sh, SliceOffsets<NQ> &o)
{
    const int lane = threadIdx.x & 31, mask = (1 << sh) - 1;
    int64_t t[NQ];
#pragma unroll
    for (int c = 0; c < NQ; ++c) t[c] = lane < CL ? tot[lane][c] : 0;
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
        const int64_t h = t[c] >> sh;
        const int l = (int)t[c] & mask;
        int64_t hi = h;
        int lo = l;
#pragma unroll
        for (int d = 1; d < kClusterMaxCtas; d <<= 1) {
            const int64_t h2 = __shfl_up_sync(0xffffffffu, hi, d);
            const int l2 = __shfl_up_sync(0xffffffffu, lo, d);
            if (lane >= d) {
                hi += h2;
                lo += l2;
            }
        }
        o.ex_hi[c] = hi - h;
        o.ex_lo[c] = lo - l;
        o.tot_hi[c] = __shfl_sync(0xffffffffu, hi, kClusterMaxCtas - 1);
        o.tot_lo[c] = __shfl_sync(0xffffffffu, lo, kClusterMaxCtas - 1);
    }
}

// The prefix in front of slice r on copy q of the ring (-1, 0, 1).
template <int NQ>
__device__ __forceinline__ void slice_base(const SliceOffsets<NQ> &o, int r, int q, int64_t (&hi)[NQ], int (&lo)[NQ])
{
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
        hi[c] = __shfl_sync(0xffffffffu, o.ex_hi[c], r) + q * o.tot_hi[c];
        lo[c] = __shfl_sync(0xffffffffu, o.ex_lo[c], r) + q * o.tot_lo[c];
    }
}

// The shifted exact window sums floor((W - own) 2^-sh) of a node from its two
// prefix entries lb, la in their slices and the slices' offsets. The entries are
// shifted one by one: their difference could pass 2^63 in slices of 512 nodes.
template <int M, int NQ>
__device__ __forceinline__ void slice_sums(const ModelParams &mp, const int64_t (&lb)[NQ], const int64_t (&la)[NQ],
                                           const int64_t (&hb)[NQ], const int64_t (&ha)[NQ], const int (&lob)[NQ],
                                           const int (&loa)[NQ], const int64_t (&qo)[NQ], int64_t (&S)[NQ])
{
    const int sh = mp.ksh, mask = (1 << sh) - 1;
    int64_t own[NQ];
    ring_own<M, NQ>(mp, qo, own);
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
        const int lo = lob[c] - loa[c] + ((int)lb[c] & mask) - ((int)la[c] & mask) - ((int)own[c] & mask);
        S[c] = hb[c] - ha[c] + (lb[c] >> sh) - (la[c] >> sh) - (own[c] >> sh) + (int64_t)(lo >> sh);
    }
}

} // namespace simk
