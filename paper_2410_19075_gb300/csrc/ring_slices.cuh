// Rings held by one thread-block cluster, every CTA a slice of consecutive nodes in
// its shared memory (RK4 in ring_cluster.cu, Dormand-Prince in ring_dp_cluster.cu):
// the slices' exact prefix offsets and the window sums across slices.
#pragma once
#include "ring_parts.cuh"

namespace simk {

// Offsets of the cluster's slices from their totals, by one warp: lane r holds the
// prefix in front of slice r as hi 2^sh + lo (ex_*), every lane the ring's total
// (tot_*).  hi is exact modulo 2^64 only (sh goes with the window, so from 1024 nodes
// on a total can be past it), which is enough for a window sum, the difference of
// two of them; the total as a value is ring_total's.
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

// The ring's exact total from its slices' totals, by one warp (every lane gets it).
template <int NQ> __device__ __forceinline__ void ring_total(const int64_t (*tot)[NQ], int CL, i128 (&sum)[NQ])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
        const int64_t t = lane < CL ? tot[lane][c] : 0;
        int64_t hi = t >> 32, lo = (int64_t)(uint32_t)t; // at most 16 terms below 2^32 each
#pragma unroll
        for (int d = kClusterMaxCtas / 2; d > 0; d >>= 1) {
            hi += __shfl_xor_sync(0xffffffffu, hi, d);
            lo += __shfl_xor_sync(0xffffffffu, lo, d);
        }
        hi = __shfl_sync(0xffffffffu, hi, 0);
        lo = __shfl_sync(0xffffffffu, lo, 0);
        sum[c] = ((i128)hi << 32) + lo;
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

// Node i (in slice rank, its prefix entry at pi) of the two-level prefix of f(y) that the
// streaming kernels read (buffer 0): lam256(i) = P(i + 1) - P(start), start the first
// node of i's 256-node sub-tile, P(start) from the entry at ps of node start - 1 in slice
// re (start = 0: ps = nullptr, re = 0).  lam256 is a difference below 2^63; the sub-tile
// starts and the total are kept exact in 128 bits.
template <int NQ>
__device__ __forceinline__ void slice_store_prefix(const RingPlan &P, const int64_t (*tot)[NQ], int CL, int i, int rank,
                                                   const int64_t *pi, int re, const int64_t *ps)
{
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
        const int64_t s = ps ? ps[c] : 0;
        uint64_t lam = (uint64_t)pi[c] - (uint64_t)s;
        for (int r = re; r < rank; ++r) lam += (uint64_t)tot[r][c];
        P.lam[0][(int64_t)i * NQ + c] = (int64_t)lam;
        if (!(i & (kSubTile - 1))) { // one prefix group (at most 32 sub-tiles): in-group offsets are the starts
            i128 start = s;
            for (int r = 0; r < re; ++r) start += tot[r][c];
            st_i128(P.ingrp[0] + c * P.nsub + (i >> kSubLog2), start);
        }
        if (i == 0) {
            i128 total = 0;
            for (int r = 0; r < CL; ++r) total += tot[r][c];
            st_i128(P.grpofs[0] + c * (P.ngroups + 1), 0);
            st_i128(P.grpofs[0] + c * (P.ngroups + 1) + 1, total);
        }
    }
}

} // namespace simk
