// Small rings resident in one thread-block cluster for a whole sim_step call.
//
// For N <= kClusterMaxNodes the stage kernels of the streaming path are
// launch-latency bound (a few CTAs per stage, four launches per RK4 step).  Here
// one cluster of up to 16 CTAs (16 SMs) runs all stages of all steps of a call:
//   * every CTA owns a contiguous slice of nodes, one per thread; their y, acc and
//     HH gates stay in registers for the whole call;
//   * after each stage every CTA builds the exact prefix lam of its slice in its own
//     shared memory (warp scans; double-buffered) and sends its slice total to
//     every CTA of the cluster (distributed shared memory); one cluster barrier
//     per stage publishes both;
//   * a node's window sum is then two 16-byte reads of lam, each in the shared memory
//     of the CTA that owns that end of the window (its address is fixed for the
//     call), plus the difference of the two slices' offsets, which every warp
//     scans from the totals itself while those reads are in flight;
//   * the order parameter of every step is recorded by one more warp of CTA 0, from
//     the exact sum of the slice totals, beside the stage that follows.
// What bounds a stage is one dependent chain: barrier, remote reads, right-hand
// side, sin/cos, scan.
// The arithmetic (grid, exact sums, right-hand sides, RK4) is the streaming
// path's, so the results are bit-for-bit the same.  At the end the cluster
// writes y, the order parameters of every step, and the streaming path's
// prefix buffers of f(y) (so that later calls may take either path).
#include <cooperative_groups.h>

#include "internal.h"
#include "ring_slices.cuh"

namespace cg = cooperative_groups;

namespace simk {

constexpr int kClusterThreadsMax = kClusterSlice + 32;

// Threads of a CTA that owns `per` nodes: one per node and the recording warp.
static __host__ __device__ constexpr int cluster_threads(int per) { return (per + 31) / 32 * 32 + 32; }

template <int NQ>
__host__ __device__ constexpr size_t cluster_smem_bytes(int per)
{
    return sizeof(int64_t) * NQ * (size_t)(2 * per); // lam, two buffers
}

template <int M>
__global__ void __launch_bounds__(kClusterThreadsMax, 1)
    ring_cluster_kernel(const RingPlan P, const StepSize h, int per, int64_t n_steps)
{
    using Mo = Model<M>;
    constexpr int D = Mo::D, NQ = Mo::NQ, NX = Mo::NX, XOFF = D - NX;
    constexpr bool KURAMOTO = M == 0 || M == 3;
    cg::cluster_group cluster = cg::this_cluster();
    cluster.barrier_arrive(); // the CTA runs: the others may store into its shared memory (publish)
    const int rank = (int)cluster.block_rank(), CL = (int)cluster.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = (int)(blockDim.x >> 5) - 1; // node warps
    const int N = (int)P.N, R = (int)P.R, sh = P.mp.ksh;
    const int i = rank * per + tid;
    const bool recorder = warp == nwarps, live = !recorder && tid < per && i < N;

    extern __shared__ __align__(16) int64_t lam[]; // [2][per][NQ]
    __shared__ __align__(16) int64_t s_tot[2][kClusterMaxCtas][NQ];
    __shared__ int64_t s_wtot[kClusterThreadsMax / 32][NQ];

    // the node's window ends: slice, copy of the ring and address of lam (buffer 0)
    int rk[2] = {0, 0}, qk[2] = {0, 0};
    const int64_t *end[2] = {lam, lam};
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        int e = side == 0 ? i + R : i - R - 1;
        if (live) {
            qk[side] = e < 0 ? -1 : (e >= N ? 1 : 0);
            e -= qk[side] * N;
            rk[side] = e / per;
            end[side] = cluster.map_shared_rank(lam, rk[side]) + (e - rk[side] * per) * NQ;
        }
    }

    double y[D] = {}, acc[D] = {}, xs[NX > 0 ? NX : 1] = {}, iext = 0.0;
    int64_t qn[NQ] = {};
    bool ok = true;
    if (live) {
#pragma unroll
        for (int v = 0; v < D; ++v) y[v] = P.y[(int64_t)v * N + i];
#pragma unroll
        for (int g = 0; g < NX; ++g) xs[g] = y[XOFF + g];
        if (M == 2 && P.node_param) iext = P.node_param[i];
        Mo::coupled_q(P.mp, y, P.F, P.lim, ok, qn);
    }

    // lam of the slice into buffer b and its total to every CTA, then the cluster barrier
    auto publish = [&](int b) {
        int64_t run[NQ];
#pragma unroll
        for (int c = 0; c < NQ; ++c) run[c] = qn[c];
        if (!recorder) {
#pragma unroll
            for (int c = 0; c < NQ; ++c) {
                run[c] = warp_incl_scan(run[c]);
                if (lane == 31) s_wtot[warp][c] = run[c];
            }
        }
        __syncthreads();
        if (live) {
            for (int w = 0; w < warp; ++w)
#pragma unroll
                for (int c = 0; c < NQ; ++c) run[c] += s_wtot[w][c];
            int64_t *o = lam + (b * per + tid) * NQ;
#pragma unroll
            for (int c = 0; c < NQ; ++c) o[c] = run[c];
        }
        if (recorder && lane < CL) {
            int64_t *o = cluster.map_shared_rank(&s_tot[b][rank][0], lane);
#pragma unroll
            for (int c = 0; c < NQ; ++c) {
                int64_t t = 0;
                for (int w = 0; w < nwarps; ++w) t += s_wtot[w][c];
                o[c] = t;
            }
        }
        cluster.sync();
    };
    auto load_end = [&](int side, int b, int64_t (&v)[NQ]) {
        const int64_t *p = end[side] + (b ? per * NQ : 0);
        if constexpr (NQ == 2) {
            const longlong2 w = *reinterpret_cast<const longlong2 *>(p);
            v[0] = w.x;
            v[1] = w.y;
        } else v[0] = *p;
    };
    auto record_order = [&](int b) { // R from buffer b's totals, by the recording warp of CTA 0
        if (!KURAMOTO || rank != 0) return;
        i128 t[NQ];
        ring_total<NQ>(s_tot[b], CL, t);
        if (lane == 0) ring_record_order(P, t[0], t[NQ - 1]);
    };

    cluster.barrier_wait(); // every CTA has started (a store into one that has not is undefined)
    // f(y) into buffer 0 (the observable of y was recorded when the state was set)
    publish(0);
    int cur = 0; // buffer holding f of the current stage input
    for (int64_t step = 0; step < n_steps; ++step) {
#pragma unroll 1
        for (int stage = 1; stage <= 4; ++stage) {
            if (!recorder) {
                int64_t lb[NQ], la[NQ], hb[NQ], ha[NQ], S[NQ];
                int lob[NQ], loa[NQ];
                load_end(0, cur, lb);
                load_end(1, cur, la);
                SliceOffsets<NQ> o;
                slice_offsets<NQ>(s_tot[cur], CL, sh, o);
                slice_base<NQ>(o, rk[0], qk[0], hb, lob);
                slice_base<NQ>(o, rk[1], qk[1], ha, loa);
                if (live) {
                    slice_sums<M, NQ>(P.mp, lb, la, hb, ha, lob, loa, qn, S);
                    double k[D], xn[D];
                    Mo::rhs_ring(P.mp, qn, S, xs, iext, k);
#pragma unroll
                    for (int v = 0; v < D; ++v) {
                        if (stage == 1) {
                            acc[v] = k[v];
                            xn[v] = y[v] + h.half * k[v];
                        } else if (stage == 4) {
                            y[v] = y[v] + h.sixth * (acc[v] + k[v]);
                            xn[v] = y[v];
                        } else {
                            acc[v] = acc[v] + 2.0 * k[v];
                            xn[v] = y[v] + (stage == 2 ? h.half : h.dt) * k[v];
                        }
                    }
#pragma unroll
                    for (int g = 0; g < NX; ++g) xs[g] = xn[XOFF + g];
                    Mo::coupled_q(P.mp, xn, P.F, P.lim, ok, qn);
                }
            } else if (KURAMOTO && stage == 1 && step > 0) { // R of y after the previous step
                record_order(cur);
            }
            cur ^= 1;
            publish(cur);
        }
    }
    if (!ok) raise_error(P.err, ERR_RANGE);

    // results: y, the last order parameter, and the streaming path's two-level prefix of f(y)
    if (recorder && n_steps > 0) record_order(cur);
    if (live) {
        const int e = (i & ~(kSubTile - 1)) - 1, re = e >= 0 ? e / per : 0;
        const int64_t *ps = e >= 0 ? cluster.map_shared_rank(lam, re) + (cur * per + e - re * per) * NQ : nullptr;
#pragma unroll
        for (int v = 0; v < D; ++v) P.y[(int64_t)v * N + i] = y[v];
        slice_store_prefix<NQ>(P, s_tot[cur], CL, i, rank, lam + (cur * per + tid) * NQ, re, ps);
    }
    cluster.sync(); // no CTA exits while others may still read its shared memory
}

static cudaLaunchConfig_t cluster_config(int cl, int per, size_t smem, cudaStream_t s, cudaLaunchAttribute *attr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cl);
    cfg.blockDim = dim3((unsigned)cluster_threads(per));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)cl;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Largest cluster of model M's kernel at its largest slice (16, or 8, the portable size)
// that the device can co-schedule, 0 if none.
template <int M> static int largest_cluster()
{
    if (cudaFuncSetAttribute(ring_cluster_kernel<M>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return 0;
    for (int cl = kClusterMaxCtas; cl >= 8; cl /= 2) {
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = cluster_config(cl, kClusterSlice, cluster_smem_bytes<Model<M>::NQ>(kClusterSlice), nullptr, &attr);
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, ring_cluster_kernel<M>, &cfg) == cudaSuccess && n >= 1) return cl;
    }
    return 0;
}

ClusterLimits cluster_limits()
{
    static PerDevice<ClusterLimits> known;
    const int dev = current_device();
    return known.get(dev, [dev] {
        ClusterLimits l;
        if (cudaDeviceGetAttribute(&l.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) l.sms = 0;
        const int rk4[4] = {largest_cluster<0>(), largest_cluster<1>(), largest_cluster<2>(), largest_cluster<3>()};
        for (int m = 0; m < 4; ++m) {
            l.rk4[m] = rk4[m];
            l.dp[m] = dp_largest_cluster(m);
        }
        cudaGetLastError(); // a query that failed answers "none"
        return l;
    });
}

int cluster_size_for(int model, int64_t N)
{
    return N <= kClusterMaxNodes ? rk4_cluster_size(cluster_limits(), model, N) : 0;
}

template <int M>
static cudaError_t launch_cluster(const RingPlan &p, double dt, int64_t n_steps, int cl, cudaStream_t s)
{
    const int per = (int)((p.N + cl - 1) / cl);
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config(cl, per, cluster_smem_bytes<Model<M>::NQ>(per), s, &attr);
    return cudaLaunchKernelEx(&cfg, ring_cluster_kernel<M>, p, step_size(dt), per, n_steps);
}

cudaError_t ring_cluster_steps(const RingPlan &p, int cl, double dt, int64_t n_steps, cudaStream_t s)
{
    cudaError_t e;
    switch (p.model) {
    case 0: e = launch_cluster<0>(p, dt, n_steps, cl, s); break;
    case 1: e = launch_cluster<1>(p, dt, n_steps, cl, s); break;
    case 2: e = launch_cluster<2>(p, dt, n_steps, cl, s); break;
    default: e = launch_cluster<3>(p, dt, n_steps, cl, s); break;
    }
    if (e == cudaSuccess) kernel_mark(s, 0);
    return e;
}

} // namespace simk
