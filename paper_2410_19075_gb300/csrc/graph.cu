// General link matrices (Section III.C) stepped with RK4 through the compressed
// form of Algorithm 2.
//
// COMPRESS (on the host, sim_api.cu) keeps a common vector V (the most frequent
// shifted row; the paper takes row 0) and, for
// every row i, a reference C_i to the difference entry D = XOR(ROL(row_i, i), V);
// EXTRACT gives row i = ROR(XOR(V, D_{C_i}), i).  So the coupling sum of node i is
//   W(i) = sum_{p in V} Q(x_{i+p}) + sum_{p in D_{C_i}} s_p Q(x_{i+p})   (indices mod N)
// with s_p = -1 where p is in V (the XOR clears that bit) and +1 elsewhere.  Here
// V is stored as runs of consecutive offsets [a, a + len), and the sum over a run
// is the difference of two entries of the exact prefix of Q in node order,
//   P(i + a + len) - P(i + a),
// the same exact fixed-point prefix the ring stage kernels build (P over the
// periodic extension).  A node therefore costs O(number of runs + size of its
// difference entry) reads instead of one per link: a ring is two runs and the
// empty entry, a periodic lattice one run per row of its window plus the
// wrapped links near the boundary.  As in the ring kernel, the exact prefix at
// the pieces the CTA's run ends fall in is computed once per CTA, so a run costs
// a node one load per end and component.  The degree of the node (its link
// count, which normalises the coupling) comes with its entry.
#include "ring_parts.cuh"

namespace simk {

// Small networks (RingPlan::flat, at most kGraphFlatSubs sub-tiles): every CTA scans
// all sub-tile totals itself (tab, the exact prefix at every sub-tile start and the
// total), so that no launch ends with the two dependent scans of its last CTAs.
// Small worlds, per RK4 step with the two-level scan and with this: 1104 nodes 43 ->
// 26 us, 20000 43 -> 28 us, 100003 54 -> 38 us.
constexpr int kGraphTab = kGraphFlatSubs + 1;

// Turn the sub-tile totals of the previous launch into tab, by the whole CTA.
template <int NQ>
__device__ __forceinline__ void graph_scan_subs(const RingPlan &P, const RingStageIO &a, i128 (*tab)[kGraphTab])
{
    constexpr int NW = kRingThreads / 32, E = kGraphFlatSubs / kRingThreads;
    __shared__ i128 s_w[NQ][NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nsub = (int)P.nsub;
    i128 v[NQ][E], ex[NQ];
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
        i128 t = 0;
#pragma unroll
        for (int u = 0; u < E; ++u) {
            const int st = tid * E + u;
            v[c][u] = st < nsub ? (i128)__ldg(a.fsub_in + c * P.nsub + st) : (i128)0;
            t += v[c][u];
        }
        const i128 x = warp_incl_scan_i128(t);
        ex[c] = x - t;
        if (lane == 31) s_w[c][warp] = x;
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < NQ; ++c) {
        for (int w = 0; w < warp; ++w) ex[c] += s_w[c][w];
#pragma unroll
        for (int u = 0; u < E; ++u) {
            const int st = tid * E + u;
            if (st <= nsub) tab[c][st] = ex[c]; // tab[nsub]: the total, by the thread one past the last
            ex[c] += v[c][u];
        }
        if (tid == kRingThreads - 1 && nsub == kGraphFlatSubs) tab[c][nsub] = ex[c];
    }
    __syncthreads();
}

// The exact prefix at the start of sub-tile st (st = nsub: the total).
template <bool FLAT>
__device__ __forceinline__ i128 graph_sub_prefix(const RingPlan &P, const RingStageIO &a, const i128 (*tab)[kGraphTab], int c,
                                                 int64_t st)
{
    if (FLAT) return tab[c][st];
    const i128 *grpofs = a.grpofs_in + c * (P.ngroups + 1);
    if (st == P.nsub) return ldg_i128(grpofs + P.ngroups);
    return ldg_i128(grpofs + (st >> kGroupLog2)) + ldg_i128(a.ingrp_in + c * P.nsub + st);
}

// Exact prefix P(pos) = sum_{m < pos} Q_m of component c on the periodic
// extension, pos in [0, 2N).
template <int NQ, bool FLAT>
__device__ __forceinline__ i128 graph_prefix_at(const RingPlan &P, const RingStageIO &a, const i128 (*tab)[kGraphTab], int c,
                                                int64_t pos)
{
    const int64_t N = P.N;
    i128 base = 0;
    if (pos >= N) {
        pos -= N;
        base = graph_sub_prefix<FLAT>(P, a, tab, c, P.nsub);
    }
    if (pos == 0) return base;
    const int64_t s = (pos - 1) >> kSubLog2;
    return base + graph_sub_prefix<FLAT>(P, a, tab, c, s) + (i128)__ldg(a.lam_in + (pos - 1) * NQ + c);
}

// Per-CTA bases of the run ends: for run r, end 2r is i + a (the run's first
// offset) and end 2r+1 is i + a + len; over the CTA's consecutive nodes each end
// covers at most three pieces (split at sub-tile starts and at N), whose exact
// prefix at the piece start is computed once, so a node needs one in-sub-tile
// prefix load per end.  Runs past kGraphSmemRuns use graph_prefix_at.
constexpr int kGraphSmemRuns = 128;
template <int NQ> struct GraphBases {
    i128 base[2 * kGraphSmemRuns][3][NQ];
    int64_t start[2 * kGraphSmemRuns][3], qn[2 * kGraphSmemRuns][3];
};

template <int NQ, bool FLAT>
__device__ __forceinline__ void graph_load_bases(const GraphPlan &G, const RingStageIO &a, const i128 (*tab)[kGraphTab],
                                                 int64_t sub, int nb, GraphBases<NQ> &B)
{
    const RingPlan &P = G.r;
    const int64_t N = P.N;
    const int64_t nvalid = N - sub * kSubTile < kSubTile ? N - sub * kSubTile : kSubTile;
    for (int e = threadIdx.x; e < 2 * nb; e += blockDim.x) {
        const int2 run = __ldg(G.runs + (e >> 1));
        const int64_t p0 = sub * kSubTile + run.x + ((e & 1) ? run.y : 0);
        const int64_t p1 = p0 + nvalid - 1; // in [0, 2N)
        int64_t p = p0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if (p > p1) {
                B.start[e][k] = INT64_MAX;
                B.qn[e][k] = 0;
                continue;
            }
            const int64_t qn = p >= N ? N : 0, pp = p - qn;
            const int64_t st = pp >> kSubLog2;
            int64_t end = ((st + 1) << kSubLog2) - 1;
            if (end > N - 1) end = N - 1;
#pragma unroll
            for (int c = 0; c < NQ; ++c) {
                B.base[e][k][c] = graph_sub_prefix<FLAT>(P, a, tab, c, st) + // pp < N: st < nsub
                                  (qn ? graph_sub_prefix<FLAT>(P, a, tab, c, P.nsub) : (i128)0);
            }
            B.start[e][k] = p;
            B.qn[e][k] = qn;
            p = end + qn + 1;
        }
    }
    __syncthreads();
}

template <int M, int NQ, bool FLAT> struct GraphGather {
    struct Pre {
        int64_t l[NQ], lp[NQ];
    };
    const GraphPlan &G;
    const RingStageIO &a;
    GraphBases<NQ> &B;
    i128 (*tab)[kGraphTab];
    int nb;      // runs with per-CTA bases
    int64_t sub; // the CTA's sub-tile
    __device__ __forceinline__ void load(int tid, int64_t i, Pre &pre) const
    {
        lam_load<NQ>(a.lam_in + i * NQ, pre.l);
#pragma unroll
        for (int c = 0; c < NQ; ++c) pre.lp[c] = 0;
        if (tid) lam_load<NQ>(a.lam_in + (i - 1) * NQ, pre.lp);
    }
    __device__ __forceinline__ void sync() const
    {
        if (FLAT) graph_scan_subs<NQ>(G.r, a, tab);
        graph_load_bases<NQ, FLAT>(G, a, tab, sub, nb, B);
    }
    template <int D>
    __device__ __forceinline__ void finish(int tid, int64_t i, const Pre &pre, const double *X, double Iext,
                                           double (&k)[D]) const
    {
        const RingPlan &P = G.r;
        const int64_t N = P.N;
        int64_t qo[NQ];
        double fo[NQ];
        i128 W[NQ];
#pragma unroll
        for (int c = 0; c < NQ; ++c) {
            qo[c] = pre.l[c] - pre.lp[c];
            fo[c] = fixed_to_double(qo[c], P.F);
            W[c] = 0;
        }
        // the common vector: runs of consecutive offsets, through the CTA's bases
        for (int r = 0; r < nb; ++r) {
            const int2 run = __ldg(G.runs + r);
            const int64_t lo = i + run.x, hi = lo + run.y;
            const int el = 2 * r, eh = 2 * r + 1;
            const int kl = (lo >= B.start[el][1]) + (lo >= B.start[el][2]);
            const int kh = (hi >= B.start[eh][1]) + (hi >= B.start[eh][2]);
            const int64_t pl = lo - B.qn[el][kl], ph = hi - B.qn[eh][kh];
            int64_t ll[NQ] = {}, lh[NQ] = {};
            if (pl & (kSubTile - 1)) lam_load<NQ>(a.lam_in + (pl - 1) * NQ, ll);
            if (ph & (kSubTile - 1)) lam_load<NQ>(a.lam_in + (ph - 1) * NQ, lh);
#pragma unroll
            for (int c = 0; c < NQ; ++c) W[c] += (B.base[eh][kh][c] - B.base[el][kl][c]) + (i128)(lh[c] - ll[c]);
        }
        for (int r = nb; r < G.nruns; ++r) {
            const int2 run = __ldg(G.runs + r); // (a, len), a + len <= N
            const int64_t lo = i + run.x, hi = lo + run.y;
#pragma unroll
            for (int c = 0; c < NQ; ++c) W[c] += graph_prefix_at<NQ, FLAT>(P, a, tab, c, hi) - graph_prefix_at<NQ, FLAT>(P, a, tab, c, lo);
        }
        // the node's difference entry: signed single links
        const int e = __ldg(G.ent + i);
        const int64_t t0 = __ldg(G.dptr + e), t1 = __ldg(G.dptr + e + 1);
        for (int64_t t = t0; t < t1; ++t) {
            const int2 d = __ldg(G.dpos + t); // (offset, sign)
            int64_t j = i + d.x;
            j -= j >= N ? N : 0;
            int64_t lj[NQ], lq[NQ] = {};
            lam_load<NQ>(a.lam_in + j * NQ, lj);
            if (j & (kSubTile - 1)) lam_load<NQ>(a.lam_in + (j - 1) * NQ, lq);
#pragma unroll
            for (int c = 0; c < NQ; ++c) W[c] += d.y > 0 ? (i128)(lj[c] - lq[c]) : -(i128)(lj[c] - lq[c]);
        }
        Model<M>::rhs(P.mp, P.F, fo, qo, W, X, Iext, k, __ldg(G.ek + e), __ldg(G.ecs + e));
    }
};

// the run loop and 128-bit window sums need more registers than the ring kernel
template <int M> struct GraphMinBlocks { static constexpr int value = 3; };
template <> struct GraphMinBlocks<2> { static constexpr int value = 2; };

template <int M, int STAGE, bool FLAT>
__global__ void __launch_bounds__(kRingThreads, GraphMinBlocks<M>::value)
    graph_stage_kernel(const GraphPlan g, const StepSize h)
{
    if (g.r.skip && *(const volatile int *)g.r.skip) return; // uniform over the launch
    constexpr int NQ = Model<M>::NQ;
    __shared__ GraphBases<NQ> s_bases;
    extern __shared__ __align__(16) i128 s_tab[]; // [NQ][kGraphTab] of a small network
    const RingStageIO a = stage_io<M, STAGE>(g.r);
    const int nb = g.nruns < kGraphSmemRuns ? g.nruns : kGraphSmemRuns;
    stage_body<M, STAGE, GraphGather<M, NQ, FLAT>, FLAT>(
        g.r, a, h, blockIdx.x,
        GraphGather<M, NQ, FLAT>{g, a, s_bases, reinterpret_cast<i128(*)[kGraphTab]>(s_tab), nb, (int64_t)blockIdx.x});
}

// static bases and dynamic table together pass 48 KB
template <int M> static cudaError_t configure()
{
    static PerDevice<cudaError_t> done;
    return done.get(current_device(), [] {
        cudaError_t err = cudaSuccess;
        const int bytes = (int)(sizeof(i128) * Model<M>::NQ * kGraphTab);
        const void *k[] = {(const void *)graph_stage_kernel<M, 1, true>, (const void *)graph_stage_kernel<M, 2, true>,
                           (const void *)graph_stage_kernel<M, 3, true>, (const void *)graph_stage_kernel<M, 4, true>};
        for (const void *f : k)
            if (err == cudaSuccess) err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        return err;
    });
}

template <int M, bool FLAT>
static cudaError_t launch_stage(int stage, const GraphPlan &g, double dt, cudaStream_t s)
{
    const cudaError_t e = FLAT ? configure<M>() : cudaSuccess;
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)g.r.nsub), block(kRingThreads);
    const size_t smem = FLAT ? sizeof(i128) * Model<M>::NQ * kGraphTab : 0;
    const StepSize h = step_size(dt);
    switch (stage) {
    case 1: graph_stage_kernel<M, 1, FLAT><<<grid, block, smem, s>>>(g, h); break;
    case 2: graph_stage_kernel<M, 2, FLAT><<<grid, block, smem, s>>>(g, h); break;
    case 3: graph_stage_kernel<M, 3, FLAT><<<grid, block, smem, s>>>(g, h); break;
    default: graph_stage_kernel<M, 4, FLAT><<<grid, block, smem, s>>>(g, h); break;
    }
    return cudaGetLastError();
}

template <int M>
static cudaError_t launch_form(int stage, const GraphPlan &g, double dt, cudaStream_t s)
{
    return g.r.flat ? launch_stage<M, true>(stage, g, dt, s) : launch_stage<M, false>(stage, g, dt, s);
}

static cudaError_t launch_any(int stage, const GraphPlan &g, double dt, cudaStream_t s)
{
    switch (g.r.model) {
    case 0: return launch_form<0>(stage, g, dt, s);
    case 1: return launch_form<1>(stage, g, dt, s);
    case 2: return launch_form<2>(stage, g, dt, s);
    default: return launch_form<3>(stage, g, dt, s);
    }
}

cudaError_t graph_rhs(const GraphPlan &g, cudaStream_t s)
{
    cudaError_t e = launch_any(1, g, 0.0, s);
    // a stage 1 on its own leaves accumulator slot 1 filled; the next RK4 step adds into it
    if (e == cudaSuccess && g.r.flat) e = ring_clear_slot(g.r, 1, s);
    return e;
}

cudaError_t graph_step(const GraphPlan &g, double dt, cudaStream_t s)
{
    for (int stage = 1; stage <= 4; ++stage) {
        const cudaError_t e = launch_any(stage, g, dt, s);
        if (e != cudaSuccess) return e;
        kernel_mark(s, 0);
    }
    return cudaSuccess;
}

} // namespace simk
