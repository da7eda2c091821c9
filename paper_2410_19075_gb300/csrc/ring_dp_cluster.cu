// Adaptive Dormand-Prince 5(4) on small rings, a whole run inside one thread-block
// cluster per ring (cluster_size.h; dp5.cu runs the others with seven launches per attempt).
//
// A batch of 1000-node rings spent seven launches per attempt on it, each reading
// every earlier slope from global memory and rebuilding the prefix hierarchy, and
// finished rings kept their share of the launches.  Here a ring's state, slopes and
// prefix stay in the shared memory of its cluster (one CTA for up to dp_slice_nodes),
// every CTA a slice of consecutive nodes as in ring_cluster.cu; the cluster takes its
// own step decisions and loops until its run is done, so rings of a batch neither
// wait for one another nor share launches.  What bounds it: the FP64 pipe (about 70
// instructions per node and attempt: tableau sums, error quotients) and, with few
// rings, one dependent chain per stage.
// The arithmetic, the order of the error sum (groups of 32 nodes, sub-tiles of 256,
// then the ring) and the controller are those of dp5.cu: the same bits, whatever
// the cluster's size.
#include <algorithm>

#include <cooperative_groups.h>

#include "dp_control.cuh"
#include "ring_slices.cuh"

namespace cg = cooperative_groups;

namespace simk {

// Threads of a CTA and nodes per thread; two CTAs per SM by registers and shared memory.
template <int M> struct DpShape { static constexpr int NT = 512, MPT = M == 0 ? 2 : 1; };
template <> struct DpShape<2> { static constexpr int NT = 256, MPT = 1; };
template <int M> constexpr bool dp_shape_fits_rule() { return DpShape<M>::NT * DpShape<M>::MPT == dp_slice(M); }
static_assert(dp_shape_fits_rule<0>() && dp_shape_fits_rule<1>() && dp_shape_fits_rule<2>() && dp_shape_fits_rule<3>(),
              "dp_slice: the kernel's slots");

template <int M> static size_t dp_cluster_smem(int per)
{
    constexpr int D = Model<M>::D, NQ = Model<M>::NQ;
    return sizeof(int64_t) * (size_t)per * (2 * NQ + 9 * D); // lam (two buffers); y, y5, k1..k7
}

// ONE: a ring in a single CTA (no offsets between slices, plain shared loads and
// barriers).
template <int M, bool ONE>
__global__ void __launch_bounds__(DpShape<M>::NT, 2)
    ring_dp_cluster_kernel(const DpPlan *__restrict__ plans, int max_attempts, int first)
{
    using Mo = Model<M>;
    constexpr int D = Mo::D, NQ = Mo::NQ, NX = Mo::NX, XOFF = D - NX, MPT = DpShape<M>::MPT;
    constexpr int NWMAX = DpShape<M>::NT / 32 * MPT;
    constexpr bool KURAMOTO = M == 0 || M == 3;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = ONE ? 0 : (int)cluster.block_rank(), CL = ONE ? 1 : (int)cluster.num_blocks();
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    const DpPlan &Q = plans[blockIdx.x / CL];
    const RingPlan &P = Q.r;
    const int N = (int)P.N, R = (int)P.R, sh = P.mp.ksh;
    const int per = ((N + CL - 1) / CL + 31) & ~31, i0 = rank * per;

    extern __shared__ __align__(16) int64_t dp_mem[];
    int64_t *lam = dp_mem;                                            // [2][per][NQ]
    double *ys = reinterpret_cast<double *>(dp_mem + 2 * NQ * per);   // [D][per]
    double *y5 = ys + D * per, *ks = y5 + D * per;                    // ks: [7][D][per], k1 first
    __shared__ __align__(16) int64_t s_tot[2][kClusterMaxCtas][NQ];
    __shared__ int64_t s_wtot[NWMAX][NQ];
    __shared__ DpCtl s_ctl;
    __shared__ int s_nhere;
    // of CTA 0: the attempt's error sums per 32 nodes, dense sums (low words, high words) and range flag
    __shared__ double s_err[kDpClusterNodes / 32];
    __shared__ unsigned long long s_out[kDpMaxOut][2][2];
    __shared__ int s_bad;
    __shared__ i128 s_sum[kDpMaxOut][2];

    if (tid == 0) s_ctl = *Q.ctl;
    __syncthreads();
    if (s_ctl.done && !first) return; // the whole cluster: every CTA reads the same word
    if constexpr (!ONE) cluster.barrier_arrive(); // the CTA runs: the others may store into its shared memory (publish)
    if (tid == 0) s_bad = 0;
    for (int q = tid; q < kDpMaxOut * 4; q += nt) (&s_out[0][0][0])[q] = 0ull;

    // own nodes l = tid + m nt of the slice; window ends as (slice, offset, copy)
    int rk[MPT][2], of[MPT][2], qk[MPT][2];
    double xs[MPT][NX > 0 ? NX : 1], iext[MPT];
    int64_t qn[MPT][NQ];
    bool ok = true;
#pragma unroll
    for (int m = 0; m < MPT; ++m) {
        const int l = tid + m * nt, i = i0 + l;
        const bool live = l < per && i < N;
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            int e = side == 0 ? i + R : i - R - 1;
            qk[m][side] = !live ? 0 : e < 0 ? -1 : (e >= N ? 1 : 0);
            e -= qk[m][side] * N;
            rk[m][side] = !ONE && live ? e / per : 0;
            of[m][side] = live ? e - rk[m][side] * per : 0;
        }
        iext[m] = M == 2 && live && P.node_param ? P.node_param[i] : 0.0;
#pragma unroll
        for (int c = 0; c < NQ; ++c) qn[m][c] = 0;
#pragma unroll
        for (int g = 0; g < NX; ++g) xs[m][g] = 0.0;
        if (live) {
#pragma unroll
            for (int v = 0; v < D; ++v) {
                ys[v * per + l] = Q.ybuf[0][(int64_t)v * N + i];
                if (!first) ks[v * per + l] = Q.k[0][(int64_t)v * N + i];
            }
        }
    }

    int cur = 0; // prefix buffer of the current stage input
    auto sync_cluster = [&]() {
        if constexpr (ONE) __syncthreads();
        else cluster.sync();
    };
    auto at = [&](auto *ptr, int r) { // ptr's object in CTA r
        if constexpr (ONE) return ptr;
        else return cluster.map_shared_rank(ptr, r);
    };
    // f(x) of the own nodes (in qn) -> their slice's prefix in buffer b and its total to every CTA
    auto publish = [&](int b) {
        int64_t run[MPT][NQ];
#pragma unroll
        for (int m = 0; m < MPT; ++m)
#pragma unroll
            for (int c = 0; c < NQ; ++c) {
                run[m][c] = warp_incl_scan(qn[m][c]);
                if (lane == 31) s_wtot[m * nw + warp][c] = run[m][c];
            }
        __syncthreads();
        int64_t tot[NQ];
#pragma unroll
        for (int c = 0; c < NQ; ++c) {
            const int64_t t = lane < MPT * nw ? s_wtot[lane][c] : 0, x = warp_incl_scan(t);
            tot[c] = __shfl_sync(0xffffffffu, x, 31);
#pragma unroll
            for (int m = 0; m < MPT; ++m) run[m][c] += __shfl_sync(0xffffffffu, x - t, m * nw + warp);
        }
#pragma unroll
        for (int m = 0; m < MPT; ++m) {
            const int l = tid + m * nt;
            if (l < per) {
                int64_t *o = lam + (b * per + l) * NQ;
#pragma unroll
                for (int c = 0; c < NQ; ++c) o[c] = run[m][c];
            }
        }
        if (tid < CL) {
            int64_t *o = at(&s_tot[b][rank][0], tid);
#pragma unroll
            for (int c = 0; c < NQ; ++c) o[c] = tot[c];
        }
        sync_cluster();
    };
    auto offsets = [&](SliceOffsets<NQ> &o) {
        if constexpr (!ONE) {
            slice_offsets<NQ>(s_tot[cur], CL, sh, o);
        } else {
#pragma unroll
            for (int c = 0; c < NQ; ++c) {
                const int64_t t = s_tot[cur][0][c];
                o.ex_hi[c] = 0;
                o.ex_lo[c] = 0;
                o.tot_hi[c] = t >> sh;
                o.tot_lo[c] = (int)t & ((1 << sh) - 1);
            }
        }
    };
    auto base = [&](const SliceOffsets<NQ> &o, int r, int q, int64_t (&hi)[NQ], int (&lo)[NQ]) {
        if constexpr (!ONE) {
            slice_base<NQ>(o, r, q, hi, lo);
        } else {
#pragma unroll
            for (int c = 0; c < NQ; ++c) {
                hi[c] = q == 0 ? 0 : (q < 0 ? -o.tot_hi[c] : o.tot_hi[c]);
                lo[c] = q == 0 ? 0 : (q < 0 ? -o.tot_lo[c] : o.tot_lo[c]);
            }
        }
    };
    // the own node m's slope at the current stage input
    auto slope = [&](const SliceOffsets<NQ> &o, int m, double (&k)[D]) {
        int64_t lb[NQ], la[NQ], hb[NQ], ha[NQ], S[NQ];
        int lob[NQ], loa[NQ];
        auto read = [&](int side, int64_t (&v)[NQ]) {
            const int64_t *ptr = at(lam, rk[m][side]) + (cur * per + of[m][side]) * NQ;
            if constexpr (NQ == 2) {
                const longlong2 w = *reinterpret_cast<const longlong2 *>(ptr);
                v[0] = w.x;
                v[1] = w.y;
            } else v[0] = *ptr;
        };
        read(0, lb);
        read(1, la);
        base(o, rk[m][0], qk[m][0], hb, lob); // shuffles between slices: every lane
        base(o, rk[m][1], qk[m][1], ha, loa);
        slice_sums<M, NQ>(P.mp, lb, la, hb, ha, lob, loa, qn[m], S);
        Mo::rhs_ring(P.mp, qn[m], S, xs[m], iext[m], k);
    };
    auto local = [&](int m, int &l) { // whether own node m exists
        l = tid + m * nt;
        return l < per && i0 + l < N;
    };
    // f(y) -> qn, its prefix
    auto publish_y = [&]() {
#pragma unroll
        for (int m = 0; m < MPT; ++m) {
            int l;
            if (!local(m, l)) continue;
            double x[D];
#pragma unroll
            for (int v = 0; v < D; ++v) x[v] = ys[v * per + l];
#pragma unroll
            for (int g = 0; g < NX; ++g) xs[m][g] = x[XOFF + g];
            Mo::coupled_q(P.mp, x, P.F, P.lim, ok, qn[m]);
        }
        if (!ok) raise_error(P.err, ERR_RANGE);
        ok = true;
        publish(cur);
    };

    if constexpr (!ONE) cluster.barrier_wait(); // every CTA has started (a store into one that has not is undefined)
    if (first) { // R(t0), k1 = f(y_n)
        publish_y();
        SliceOffsets<NQ> o;
        offsets(o);
        if (KURAMOTO && rank == 0 && warp == 0 && P.obs) {
            i128 t[NQ];
            ring_total<NQ>(s_tot[cur], CL, t);
            if (lane == 0) ring_record_order(P, t[0], t[NQ - 1]);
        }
        if (!s_ctl.done) {
#pragma unroll
            for (int m = 0; m < MPT; ++m) {
                int l;
                const bool live = local(m, l);
                double k[D];
                slope(o, m, k);
                if (live)
#pragma unroll
                    for (int v = 0; v < D; ++v) ks[v * per + l] = k[v];
            }
        }
        cur ^= 1;
    }
    sync_cluster(); // s_out, s_bad zeroed and every own load done before the first attempt

    for (int att = 0; att < max_attempts && !s_ctl.done; ++att) {
        const double h = s_ctl.h_att, t = s_ctl.t;
        if (tid == 0) { // dense outputs inside (t, t + h]
            int n = 0;
            if (KURAMOTO && s_ctl.out_dt > 0.0) {
                while (n < kDpMaxOut && s_ctl.next_out + n <= s_ctl.n_out) {
                    const double to = s_ctl.t0 + (double)(s_ctl.next_out + n) * s_ctl.out_dt;
                    if (!s_ctl.last && to > t + h) break;
                    ++n;
                }
            }
            s_nhere = n;
        }
        // s = 1: the input of stage 2 from the kept k1; s = 2..6: k_s and the input of
        // stage s + 1 (x7 is the candidate y_{n+1}); s = 7: k7
#pragma unroll 1
        for (int s = 1; s <= 7; ++s) {
            SliceOffsets<NQ> o;
            if (s > 1) offsets(o);
#pragma unroll
            for (int m = 0; m < MPT; ++m) {
                int l;
                const bool live = local(m, l);
                double k[D];
                if (s > 1) slope(o, m, k);
                if (!live) continue;
                if (s > 1)
#pragma unroll
                    for (int v = 0; v < D; ++v) ks[((s - 1) * D + v) * per + l] = k[v];
                if (s == 7) continue;
                double x[D];
#pragma unroll
                for (int v = 0; v < D; ++v) {
                    const double *kv = ks + v * per + l;
                    double acc = s == 1 ? c_dp_a[1][0] * kv[0]
                                        : dp_sum2(c_dp_a[s][0], kv[0], c_dp_a[s][1], kv[D * per]);
#pragma unroll 1
                    for (int j = 2; j < s; ++j) acc = fma(c_dp_a[s][j], kv[j * D * per], acc);
                    x[v] = fma(h, acc, ys[v * per + l]);
                    if (s == 6) y5[v * per + l] = x[v];
                }
#pragma unroll
                for (int g = 0; g < NX; ++g) xs[m][g] = x[XOFF + g];
                Mo::coupled_q(P.mp, x, P.F, P.lim, ok, qn[m]);
            }
            if (s < 7) {
                if (s > 1) cur ^= 1;
                publish(cur);
            }
        }
        // error and dense-output sums
        const int n_here = s_nhere;
        const double atol = s_ctl.atol, rtol = s_ctl.rtol;
        double *err0 = at(s_err, 0);
#pragma unroll
        for (int m = 0; m < MPT; ++m) {
            int l;
            const bool live = local(m, l);
            double err = 0.0;
            if (live) {
#pragma unroll
                for (int v = 0; v < D; ++v) {
                    const double *kv = ks + v * per + l;
                    double e = dp_sum2(c_dp_e[0], kv[0], c_dp_e[2], kv[2 * D * per]);
#pragma unroll
                    for (int j = 3; j <= 6; ++j) e = fma(c_dp_e[j], kv[j * D * per], e);
                    e *= h;
                    const double sc = atol + rtol * fmax(fabs(ys[v * per + l]), fabs(y5[v * per + l]));
                    const double r = e / sc;
                    err += r * r;
                }
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) err += __shfl_xor_sync(0xffffffffu, err, d);
            if (lane == 0 && l < per && i0 + l < N) err0[(i0 + l) >> 5] = err;
        }
        for (int q = 0; q < n_here; ++q) {
            long long ss = 0, cc = 0;
#pragma unroll
            for (int m = 0; m < MPT; ++m) {
                int l;
                if (!local(m, l)) continue;
                const double to = s_ctl.t0 + (double)(s_ctl.next_out + q) * s_ctl.out_dt;
                double th = (to - t) / h;
                th = th > 1.0 ? 1.0 : th;
                const double a0 = ys[l], a1 = y5[l], f0 = ks[l], f1 = ks[6 * D * per + l];
                const double ph = dp_hermite(th, h, a0, a1, f0, f1);
                int64_t s62, c62;
                fixed_sincos(ph, P.mp.tab, s62, c62, ok);
                ss += q62_to(s62, P.F);
                cc += q62_to(c62, P.F);
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) {
                ss += __shfl_xor_sync(0xffffffffu, ss, d);
                cc += __shfl_xor_sync(0xffffffffu, cc, d);
            }
            if (lane == 0) { // exact in any order: low words and signed high words apart
                unsigned long long *o0 = at(&s_out[q][0][0], 0);
                atomicAdd(o0 + 0, (unsigned long long)ss & 0xffffffffull);
                atomicAdd(o0 + 1, (unsigned long long)(ss >> 32));
                atomicAdd(o0 + 2, (unsigned long long)cc & 0xffffffffull);
                atomicAdd(o0 + 3, (unsigned long long)(cc >> 32));
            }
        }
        if (!ok) atomicOr(at(&s_bad, 0), 1);
        ok = true;
        sync_cluster();
        if (rank == 0 && warp == 0) { // the decision
            double a = 0.0;
            const int ng = (N + 31) >> 5;
#pragma unroll
            for (int w = 0; w < 8; ++w)
                if (lane * 8 + w < ng) a += s_err[lane * 8 + w];
            for (int d = 16; d > 0; d >>= 1) a += __shfl_xor_sync(0xffffffffu, a, d);
            if (lane < n_here)
                for (int c = 0; c < 2; ++c) {
                    s_sum[lane][c] = (i128)s_out[lane][c][0] + ((i128)(long long)s_out[lane][c][1] << 32);
                    s_out[lane][c][0] = s_out[lane][c][1] = 0ull;
                }
            __syncwarp();
            if (lane == 0) {
                if (s_bad) s_ctl.bad = 1;
                s_bad = 0;
                dp_decide_ctl(&s_ctl, Q.remaining, a, (int64_t)D * N, n_here, s_sum,
                              DpRecord{P.obs, P.obs_cap, P.obs_ctr, P.F, P.N});
            }
            __syncwarp();
            if (!ONE && lane > 0 && lane < CL) *at(&s_ctl, lane) = s_ctl;
        }
        sync_cluster();
        if (s_ctl.acc_flag) { // y <- y_{n+1}, k1 <- k7
#pragma unroll
            for (int m = 0; m < MPT; ++m) {
                int l;
                if (!local(m, l)) continue;
#pragma unroll
                for (int v = 0; v < D; ++v) {
                    ys[v * per + l] = y5[v * per + l];
                    ks[v * per + l] = ks[(6 * D + v) * per + l];
                }
            }
        }
    }

    // results: y, k1 and the controls for a next launch, and the two-level prefix of
    // f(y) the other kernels read (buffer 0), as in ring_cluster.cu
    publish_y();
#pragma unroll
    for (int m = 0; m < MPT; ++m) {
        int l;
        if (!local(m, l)) continue;
        const int i = i0 + l, e = (i & ~(kSubTile - 1)) - 1, re = e >= 0 ? e / per : 0;
        const int64_t *ps = e >= 0 ? at(lam, re) + (cur * per + e - re * per) * NQ : nullptr;
#pragma unroll
        for (int v = 0; v < D; ++v) {
            Q.ybuf[0][(int64_t)v * N + i] = ys[v * per + l];
            Q.k[0][(int64_t)v * N + i] = ks[v * per + l];
        }
        slice_store_prefix<NQ>(P, s_tot[cur], CL, i, rank, lam + (cur * per + l) * NQ, re, ps);
    }
    if (rank == 0 && tid == 0) {
        s_ctl.cur = 0; // y_n and k1 are in the first buffers
        *Q.ctl = s_ctl;
    }
    sync_cluster(); // no CTA exits while others may still read its shared memory
}

template <int M, bool ONE> static cudaError_t configure_shape()
{
    cudaError_t e = cudaFuncSetAttribute(ring_dp_cluster_kernel<M, ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)dp_cluster_smem<M>(dp_slice(M)));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(ring_dp_cluster_kernel<M, ONE>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

template <int M>
static cudaLaunchConfig_t shape_config(int n, int cl, int per, cudaStream_t s, cudaLaunchAttribute *attr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(cl * n));
    cfg.blockDim = dim3((unsigned)std::min(DpShape<M>::NT, per));
    cfg.dynamicSmemBytes = dp_cluster_smem<M>(per);
    cfg.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)cl;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Attributes of model M's kernels on the current device, and the largest cluster at a
// full slice it can co-schedule (0: none).
template <int M> static int largest_cluster()
{
    if (configure_shape<M, true>() != cudaSuccess || configure_shape<M, false>() != cudaSuccess) return 0;
    for (int cl = kClusterMaxCtas; cl >= 1; cl /= 2) {
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = shape_config<M>(1, cl, dp_slice(M), nullptr, &attr);
        int n = 0;
        const cudaError_t e = cl > 1 ? cudaOccupancyMaxActiveClusters(&n, ring_dp_cluster_kernel<M, false>, &cfg)
                                     : cudaOccupancyMaxActiveClusters(&n, ring_dp_cluster_kernel<M, true>, &cfg);
        if (e == cudaSuccess && n >= 1) return cl;
    }
    return 0;
}
int dp_largest_cluster(int model)
{
    switch (model) {
    case 0: return largest_cluster<0>();
    case 1: return largest_cluster<1>();
    case 2: return largest_cluster<2>();
    default: return largest_cluster<3>();
    }
}

template <int M, bool ONE>
static cudaError_t launch_shape(const DpPlan *plans, int n, int cl, int64_t n_max, int max_attempts, int first, cudaStream_t s)
{
    const int per = (int)(((n_max + cl - 1) / cl + 31) / 32 * 32); // of the largest ring of the launch
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = shape_config<M>(n, cl, per, s, &attr);
    return cudaLaunchKernelEx(&cfg, ring_dp_cluster_kernel<M, ONE>, plans, max_attempts, first);
}

template <int M>
static cudaError_t launch_m(const DpPlan *plans, int n, int cl, int64_t n_max, int max_attempts, int first, cudaStream_t s)
{
    return cl == 1 ? launch_shape<M, true>(plans, n, cl, n_max, max_attempts, first, s)
                   : launch_shape<M, false>(plans, n, cl, n_max, max_attempts, first, s);
}

cudaError_t dp_cluster_launch(int model, const DpPlan *plans, int n, int cl, int64_t n_max, int max_attempts, int first,
                              cudaStream_t s)
{
    switch (model) {
    case 0: return launch_m<0>(plans, n, cl, n_max, max_attempts, first, s);
    case 1: return launch_m<1>(plans, n, cl, n_max, max_attempts, first, s);
    case 2: return launch_m<2>(plans, n, cl, n_max, max_attempts, first, s);
    default: return launch_m<3>(plans, n, cl, n_max, max_attempts, first, s);
    }
}

} // namespace simk
