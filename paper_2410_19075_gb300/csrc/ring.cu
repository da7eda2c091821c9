// Ring topology: one fused kernel per RK4 stage.
//
// Stage s (s = 1..4) of node i, in one pass over the ring (Section IV 1D
// networks; the per-node right-hand side of Algorithm 1):
//   a3  window sums   W(i) = P(i+R+1) - P(i-R), P(p) = sum_{j<p} Q(f_j) over the
//                     periodic extension, read from the exact prefix arrays the
//                     previous kernel wrote (two shifted reads; the quantities
//                     of a node interleaved, one 16-byte load per read);
//   a4  right-hand side k_s(i) from W(i) and the node's own stage input;
//   a5  RK4 accumulate acc += b_s k_s (stage 4: y <- y + dt/6 (acc + k_4));
//   a1  next stage input x_{s+1} = y + c_{s+1} dt k_s;
//   a2  coupled quantity f(x_{s+1}), its exact prefix inside each 256-node
//       sub-tile (one CTA), and, without any CTA waiting for another, the exact
//       prefix at every sub-tile start: the last CTA to finish in each group of
//       64 sub-tiles scans that group, and the last group scans the groups; or,
//       for rings of at most 128 groups (one-pass prefix, ring_parts.cuh), the
//       sub-tile totals and group accumulators the next kernel sums itself;
//   a6  (stage 4) the Kuramoto order parameter of y_{n+1} from the global totals.
// The prologue kernel does a1/a2/a6 for the initial state.  The Kuramoto and
// FHN rings run ring_stage_kernel2 (two adjacent nodes per thread) unless the
// autotuner chose ring_stage_kernel (one node per thread), which HH always
// runs.  The building blocks are in ring_parts.cuh.
#include "ring_parts.cuh"

namespace simk {

// Ring window in three phases.  load(): the node's own prefix entries and those
// at its window ends.  sync(): the bases become visible.  finish(): the shifted
// exact window sums and the node's slope.
template <int M, int NQ> struct RingGather {
    struct Pre {
        int64_t l[NQ], lp[NQ], lb[NQ], la[NQ];
    };
    const RingPlan &P;
    const int64_t *lam_in;
    const RingBases<NQ> &B;
    int64_t sub;
    __device__ __forceinline__ void load(int tid, int64_t i, Pre &pre) const
    {
        lam_load<NQ>(lam_in + i * NQ, pre.l);
#pragma unroll
        for (int c = 0; c < NQ; ++c) pre.lp[c] = 0;
        if (tid) lam_load<NQ>(lam_in + (i - 1) * NQ, pre.lp);
        lam_load_end<NQ>(ring_end<NQ>(P, lam_in, sub, 0), tid, pre.lb);
        lam_load_end<NQ>(ring_end<NQ>(P, lam_in, sub, 1), tid, pre.la);
    }
    __device__ __forceinline__ void sync() const { __syncthreads(); }
    template <int D>
    __device__ __forceinline__ void finish(int tid, int64_t, const Pre &pre, const double *X, double Iext,
                                           double (&k)[D]) const
    {
        int64_t qo[NQ], own[NQ], S[NQ];
#pragma unroll
        for (int c = 0; c < NQ; ++c) qo[c] = pre.l[c] - pre.lp[c];
        ring_own<M, NQ>(P.mp, qo, own);
        ring_sums<NQ>(B, tid, P.mp.ksh, pre.lb, pre.la, own, S);
        Model<M>::rhs_ring(P.mp, qo, S, X, Iext, k);
    }
};

// One 256-node sub-tile `sub` of ring P, one node per thread (the whole CTA).
// FLAT_OK: the plain kernel, which may run the one-pass prefix (batched members
// always keep the two-level scan).
template <int M, int STAGE, bool FLAT_OK>
__device__ __forceinline__ void ring_stage_body(const RingPlan &P, const RingStageIO &a, const StepSize &h,
                                                int64_t sub)
{
    constexpr int NQ = Model<M>::NQ;
    __shared__ RingBases<NQ> s_bases;
    if (STAGE > 0) {
        if (FLAT_OK && P.flat) ring_flat_bases<NQ>(P, a.fsub_in, a.facc_in, sub, s_bases);
        else ring_compute_bases<NQ>(P, a.ingrp_in, a.grpofs_in, sub, s_bases);
    }
    stage_body<M, STAGE, RingGather<M, NQ>, FLAT_OK>(P, a, h, sub, RingGather<M, NQ>{P, a.lam_in, s_bases, sub});
}

// Two adjacent nodes per thread, 128 threads per 256-node sub-tile: two
// independent right-hand sides per thread and one warp scan per node pair.  The
// same integers and FP64 expressions as ring_stage_body, so the same bits.
constexpr int kRing2Threads = kSubTile / 2;
// Resident CTAs per SM the registers are sized for: 8 (64 registers), for Kuramoto with
// inertia 7 (72), which spills less.  Its RK4 steps with 8 / 7 / 6 per SM, in us: 26.2 / 24.2 /
// 24.2 at 50000 nodes, 64.5 / 63.4 / 71.9 at 5 10^5, 539 / 533 / 570 at 5 10^6, 512 rings of
// 1000 80.7 / 80.3 / 87.6; but 42.7 / 51.9 / 52.1 at 3 10^5, where 8 make one wave of what takes
// two with 7 (ring2_in_one_wave).  The other models lose 2% with 7.
template <int M> struct Ring2MinBlocks { static constexpr int value = 8; };
template <> struct Ring2MinBlocks<3> { static constexpr int value = 7; };

template <int M, int STAGE>
__device__ __forceinline__ void ring_stage_body2(const RingPlan &P, const RingStageIO &a, const StepSize &h,
                                                 int64_t sub)
{
    using Mo = Model<M>;
    constexpr int D = Mo::D, NQ = Mo::NQ, NX = Mo::NX;
    constexpr int XOFF = D - NX;
    __shared__ RingBases<NQ> s_bases;
    const int tid = threadIdx.x, l0 = 2 * tid;
    const int64_t N = P.N, s0 = sub * kSubTile;
    const int nv = (int)(N - s0 < kSubTile ? N - s0 : kSubTile); // nodes of the sub-tile
    const bool flat = P.flat != 0;
    if (STAGE > 0) {
        if (flat) ring_flat_bases<NQ>(P, a.fsub_in, a.facc_in, sub, s_bases);
        else ring_compute_bases<NQ>(P, a.ingrp_in, a.grpofs_in, sub, s_bases);
    }

    int64_t ln[2][NQ], lp[NQ], lb[2][NQ], la[2][NQ];
    double yv[2][D], av[2][D], X[2][NX > 0 ? NX : 1];
    const double *ys = P.y + s0;
    double *accs = P.acc + s0;
    if (STAGE > 0) {
        const int64_t *lam = a.lam_in + s0 * NQ;
        const RingEnd<NQ> eb = ring_end<NQ>(P, a.lam_in, sub, 0), ea = ring_end<NQ>(P, a.lam_in, sub, 1);
#pragma unroll
        for (int c = 0; c < NQ; ++c) lp[c] = 0;
        if (tid && l0 < nv) lam_load<NQ>(lam + (l0 - 1) * NQ, lp);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int l = l0 + u;
            if (l < nv) {
                lam_load<NQ>(lam + l * NQ, ln[u]);
                lam_load_end<NQ>(eb, l, lb[u]);
                lam_load_end<NQ>(ea, l, la[u]);
#pragma unroll
                for (int v = 0; v < D; ++v) {
                    yv[u][v] = ys[v * N + l];
                    av[u][v] = STAGE >= 2 ? accs[v * N + l] : 0.0;
                }
#pragma unroll
                for (int g = 0; g < NX; ++g) X[u][g] = a.x_in[s0 + g * N + l];
            }
        }
        __syncthreads();
    }

    int64_t qv[2][NQ];
    bool ok = true;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int l = l0 + u;
#pragma unroll
        for (int c = 0; c < NQ; ++c) qv[u][c] = 0;
        if (l >= nv) continue;
        double xn[D];
        if (STAGE == 0) {
#pragma unroll
            for (int v = 0; v < D; ++v) xn[v] = ys[v * N + l];
        } else {
            int64_t qo[NQ], own[NQ], S[NQ];
#pragma unroll
            for (int c = 0; c < NQ; ++c) qo[c] = ln[u][c] - (u == 0 ? lp[c] : ln[0][c]);
            ring_own<M, NQ>(P.mp, qo, own);
            ring_sums<NQ>(s_bases, l, P.mp.ksh, lb[u], la[u], own, S);
            double k[D];
            Mo::rhs_ring(P.mp, qo, S, X[u], 0.0, k);
#pragma unroll
            for (int v = 0; v < D; ++v) {
                if (STAGE == 1) {
                    accs[v * N + l] = k[v];
                    xn[v] = yv[u][v] + h.half * k[v];
                } else if (STAGE == 2) {
                    accs[v * N + l] = av[u][v] + 2.0 * k[v];
                    xn[v] = yv[u][v] + h.half * k[v];
                } else if (STAGE == 3) {
                    accs[v * N + l] = av[u][v] + 2.0 * k[v];
                    xn[v] = yv[u][v] + h.dt * k[v];
                } else {
                    const double yn = yv[u][v] + h.sixth * (av[u][v] + k[v]);
                    P.y[s0 + v * N + l] = yn;
                    xn[v] = yn;
                }
            }
            if (NX > 0 && STAGE >= 1 && STAGE <= 3) {
#pragma unroll
                for (int g = 0; g < NX; ++g) a.x_out[s0 + g * N + l] = xn[XOFF + g];
            }
        }
        Mo::coupled_q(P.mp, xn, P.F, P.lim, ok, qv[u]);
    }
    if (!ok) raise_error(P.err, ERR_RANGE);
    // the prologue writes both prefix forms (a later kernel of either kind may read it)
    ring_prefix_tail_n<NQ, 2, (M == 0 || M == 3) && (STAGE == 0 || STAGE == 4), STAGE == 4>(
        P, a.lam_out, a.ingrp_out, a.grpofs_out, sub, s0 + l0, qv, flat, STAGE == 0 || !flat, a.fsub_out, a.facc_out,
        a.facc_zero);
}

template <int M, int STAGE, int CTAS = Ring2MinBlocks<M>::value>
__global__ void __launch_bounds__(kRing2Threads, CTAS) ring_stage_kernel2(const RingPlan p, const StepSize h)
{
    if (p.skip && *(const volatile int *)p.skip) return; // uniform over the launch
    ring_stage_body2<M, STAGE>(p, stage_io<M, STAGE>(p), h, blockIdx.x);
}

// Plain path: one ring, one sub-tile per CTA.
template <int M, int STAGE>
__global__ void __launch_bounds__(kRingThreads, MinBlocks<M>::value) ring_stage_kernel(const RingPlan p, const StepSize h)
{
    if (p.skip && *(const volatile int *)p.skip) return; // uniform over the launch
    ring_stage_body<M, STAGE, true>(p, stage_io<M, STAGE>(p), h, blockIdx.x);
}

// Batched path: CTA b works on sub-tile b - item_base[inst] of ring inst =
// inst_of_item[b]; every ring keeps its own exact prefix hierarchy.  A ring whose
// step budget (steps_left) is used up is skipped whole, so its arrival counters
// stay consistent.  The plan is staged in shared memory: read from global memory
// where each field is first used, behind the budget's own dependent load, warps
// waited on loads five times as long as a single ring's kernel does, and 512 rings
// of 100 to 50,000 nodes took 543 us per RK4 step, here 465.
template <int M, int STAGE>
__global__ void __launch_bounds__(kRingThreads, MinBlocks<M>::value)
    ring_batch_stage_kernel(const RingPlan *__restrict__ plans, const int *__restrict__ inst_of_item,
                            const int64_t *__restrict__ item_base, const volatile long long *steps_left,
                            const StepSize h)
{
    __shared__ __align__(16) unsigned char plan_mem[sizeof(RingPlan)];
    RingPlan &p = *reinterpret_cast<RingPlan *>(plan_mem);
    const int inst = inst_of_item[blockIdx.x];
    const int64_t sub = (int64_t)blockIdx.x - item_base[inst];
    const long long left = steps_left[inst]; // loaded together with the plan
    stage_plan(p, plans + inst);
    if (left <= 0) return;
    ring_stage_body<M, STAGE, false>(p, stage_io<M, STAGE>(p), h, sub);
}

// The same with two adjacent nodes per thread (ring_stage_body2).
template <int M, int STAGE>
__global__ void __launch_bounds__(kRing2Threads, Ring2MinBlocks<M>::value)
    ring_batch_stage_kernel2(const RingPlan *__restrict__ plans, const int *__restrict__ inst_of_item,
                             const int64_t *__restrict__ item_base, const volatile long long *steps_left,
                             const StepSize h)
{
    __shared__ __align__(16) unsigned char plan_mem[sizeof(RingPlan)];
    RingPlan &p = *reinterpret_cast<RingPlan *>(plan_mem);
    const int inst = inst_of_item[blockIdx.x];
    const int64_t sub = (int64_t)blockIdx.x - item_base[inst];
    const long long left = steps_left[inst]; // loaded together with the plan
    stage_plan(p, plans + inst);
    if (left <= 0) return;
    ring_stage_body2<M, STAGE>(p, stage_io<M, STAGE>(p), h, sub);
}

// Whether all sub-tiles of a ring are resident at once with 8 CTAs per SM and not with
// the fewer its model is compiled for.
template <int M> static bool ring2_in_one_wave(const RingPlan &p)
{
    if (Ring2MinBlocks<M>::value >= 8) return false;
    static PerDevice<int> sms;
    const int dev = current_device(), n = sms.get(dev, [dev] {
        int v = 0;
        return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess ? v : 0;
    });
    return p.nsub > Ring2MinBlocks<M>::value * n && p.nsub <= 8 * n;
}

template <int M, int CTAS> static void launch_stage2(int stage, const RingPlan &p, const StepSize &h, cudaStream_t s)
{
    const dim3 grid((unsigned)p.nsub), block(kRing2Threads);
    switch (stage) {
    case 0: ring_stage_kernel2<M, 0><<<grid, block, 0, s>>>(p, h); break;
    case 1: ring_stage_kernel2<M, 1, CTAS><<<grid, block, 0, s>>>(p, h); break;
    case 2: ring_stage_kernel2<M, 2, CTAS><<<grid, block, 0, s>>>(p, h); break;
    case 3: ring_stage_kernel2<M, 3, CTAS><<<grid, block, 0, s>>>(p, h); break;
    default: ring_stage_kernel2<M, 4, CTAS><<<grid, block, 0, s>>>(p, h); break;
    }
}

// The kernel variant is the plan's (p.npt, from sim_create or the autotuner):
// two nodes per thread (128 threads per sub-tile) or one (256).
template <int M>
static cudaError_t launch_stage(int stage, const RingPlan &p, double dt, cudaStream_t s)
{
    const dim3 grid((unsigned)p.nsub), block(kRingThreads);
    if constexpr (M != 2) {
        if (p.npt == 2) {
            if (ring2_in_one_wave<M>(p)) launch_stage2<M, 8>(stage, p, step_size(dt), s);
            else launch_stage2<M, Ring2MinBlocks<M>::value>(stage, p, step_size(dt), s);
            return cudaGetLastError();
        }
    }
    switch (stage) {
    case 0: ring_stage_kernel<M, 0><<<grid, block, 0, s>>>(p, step_size(dt)); break;
    case 1: ring_stage_kernel<M, 1><<<grid, block, 0, s>>>(p, step_size(dt)); break;
    case 2: ring_stage_kernel<M, 2><<<grid, block, 0, s>>>(p, step_size(dt)); break;
    case 3: ring_stage_kernel<M, 3><<<grid, block, 0, s>>>(p, step_size(dt)); break;
    default: ring_stage_kernel<M, 4><<<grid, block, 0, s>>>(p, step_size(dt)); break;
    }
    return cudaGetLastError();
}

static cudaError_t launch_any(int stage, const RingPlan &p, double dt, cudaStream_t s)
{
    switch (p.model) {
    case 0: return launch_stage<0>(stage, p, dt, s);
    case 1: return launch_stage<1>(stage, p, dt, s);
    case 2: return launch_stage<2>(stage, p, dt, s);
    default: return launch_stage<3>(stage, p, dt, s);
    }
}

template <int M>
static cudaError_t launch_batch_stage(int stage, const RingBatchGroup &g, double dt, cudaStream_t s)
{
    const dim3 grid((unsigned)g.n_items), block(kRingThreads);
    const StepSize h = step_size(dt);
    if constexpr (M != 2) {
        if (g.npt == 2) {
            const dim3 block2(kRing2Threads);
            switch (stage) {
            case 1: ring_batch_stage_kernel2<M, 1><<<grid, block2, 0, s>>>(g.plans, g.inst_of_item, g.item_base, g.steps_left, h); break;
            case 2: ring_batch_stage_kernel2<M, 2><<<grid, block2, 0, s>>>(g.plans, g.inst_of_item, g.item_base, g.steps_left, h); break;
            case 3: ring_batch_stage_kernel2<M, 3><<<grid, block2, 0, s>>>(g.plans, g.inst_of_item, g.item_base, g.steps_left, h); break;
            default: ring_batch_stage_kernel2<M, 4><<<grid, block2, 0, s>>>(g.plans, g.inst_of_item, g.item_base, g.steps_left, h); break;
            }
            return cudaGetLastError();
        }
    }
    switch (stage) {
    case 1: ring_batch_stage_kernel<M, 1><<<grid, block, 0, s>>>(g.plans, g.inst_of_item, g.item_base, g.steps_left, h); break;
    case 2: ring_batch_stage_kernel<M, 2><<<grid, block, 0, s>>>(g.plans, g.inst_of_item, g.item_base, g.steps_left, h); break;
    case 3: ring_batch_stage_kernel<M, 3><<<grid, block, 0, s>>>(g.plans, g.inst_of_item, g.item_base, g.steps_left, h); break;
    default: ring_batch_stage_kernel<M, 4><<<grid, block, 0, s>>>(g.plans, g.inst_of_item, g.item_base, g.steps_left, h); break;
    }
    return cudaGetLastError();
}

cudaError_t ring_batch_step(const RingBatchGroup &g, double dt, cudaStream_t s)
{
    if (g.n_items == 0) return cudaSuccess;
    for (int stage = 1; stage <= 4; ++stage) {
        cudaError_t e;
        switch (g.model) {
        case 0: e = launch_batch_stage<0>(stage, g, dt, s); break;
        case 1: e = launch_batch_stage<1>(stage, g, dt, s); break;
        case 2: e = launch_batch_stage<2>(stage, g, dt, s); break;
        default: e = launch_batch_stage<3>(stage, g, dt, s); break;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static size_t flat_slot_bytes(const RingPlan &p)
{
    return sizeof(unsigned) * 4 * (size_t)(p.model == 2 ? Model<2>::NQ : Model<0>::NQ) * (size_t)p.ngroups;
}

cudaError_t ring_prologue(const RingPlan &p, cudaStream_t s)
{
    if (p.flat) { // the four accumulator slots are contiguous; slot 0 must start from zero
        const cudaError_t e = cudaMemsetAsync(p.facc[0], 0, 4 * flat_slot_bytes(p), s);
        if (e != cudaSuccess) return e;
    }
    return launch_any(0, p, 0.0, s);
}

cudaError_t ring_clear_slot(const RingPlan &p, int slot, cudaStream_t s)
{
    return cudaMemsetAsync(p.facc[slot], 0, flat_slot_bytes(p), s);
}

cudaError_t ring_rhs(const RingPlan &p, cudaStream_t s)
{
    cudaError_t e = launch_any(1, p, 0.0, s);
    // a stage 1 on its own leaves slot 1 filled; the next RK4 step adds into it
    if (e == cudaSuccess && p.flat) e = ring_clear_slot(p, 1, s);
    return e;
}

cudaError_t ring_step(const RingPlan &p, double dt, cudaStream_t s)
{
    for (int stage = 1; stage <= 4; ++stage) {
        const cudaError_t e = launch_any(stage, p, dt, s);
        if (e != cudaSuccess) return e;
        kernel_mark(s, 0);
    }
    return cudaSuccess;
}

} // namespace simk
