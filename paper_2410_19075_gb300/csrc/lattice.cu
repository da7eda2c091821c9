// Periodic lattices of Kuramoto nodes (with or without inertia), Section IV:
//   cube  N1^3 nodes, index k N1^2 + j N1 + i, the (2P+1)^3 box around a node;
//   ball  N1^3 nodes, the sphere dx^2 + dy^2 + dz^2 <= P^2 (3D networks);
//   disk  N1^2 nodes, index j N1 + i, the circle dx^2 + dy^2 <= P^2 (2D networks).
// f = (sin, cos) of the stage-input phase, rounded onto the grid 2^-F (F chosen
// so that a full window sum fits in int64), so every window sum is exact
// integer arithmetic and the node's right-hand side needs one cross product of
// the sums with its own (sin, cos).  The ball and disk rotate every node's
// quantity by -alpha in the x pass (lattice_rotated_q); the cube keeps its sums
// unrotated and turns the node's own phase by +alpha (own_phase_turned).
//
// Cube, per RK4 stage (the box is separable):
//   x pass  SX(i,j,k)  = sum_{|dx|<=P} Q(f(i+dx,j,k))      (row prefix in shared memory)
//   y pass  SXY(i,j,k) = sum_{|dy|<=P} SX(i,j+dy,k)        (column prefix in a tile)
//   z pass  W(i,j,k)   = sum_{|dz|<=P} SXY(i,j,k+dz)       (column prefix in a tile)
//           and the coupling term; the node pass then runs the right-hand side,
//           the RK4 update, the next (sin, cos) and the next stage's x pass.
//           Both sums are (sin, cos) pairs: one address, one wrap test and one
//           16-byte shared access serve the two components (two separate arrays
//           took 172 instructions per node in the y pass of a 101^3 cube, pairs
//           122).  Batched cubes run the same passes, one launch for all members.
// Ball and disk, per RK4 stage:
//   x pass  balls of P >= 5: for every half-width w = 0..P the x-window sums S_w(i) of
//           Q(f) along every row, sin and cos interleaved; otherwise, and when those
//           P+1 arrays would exceed the memory budget (or SIM_FLAG_LOW_MEMORY), the
//           inclusive row prefix E(x) extended periodically by P + 1 entries on the
//           left and P on the right (wrapping int64);
//   gather  W = sum over the chords of the window, one per (dy, dz) (ball) or dy
//           (disk): the row segment |dx| <= w = floor(sqrt(P^2 - dy^2 - dz^2)),
//           read as S_w (one 16-byte load) or E(i + w) - E(i - w - 1) (two),
//           O(P^2) resp. O(P) reads per node, up to four neighbouring nodes per thread
//           sharing the reads their windows have in common, fused with the right-hand side
//           and RK4 update.
#include <algorithm>

#include "internal.h"

namespace simk {

constexpr int kRowWarpsMax = 8;       // x pass: one warp per row
constexpr int kGatherThreads = 128;   // ball/disk gather: a block of rows x planes of nodes per thread
constexpr int kGatherOps = 512;       // ball/disk gather: reads of the window held in shared memory at a time
constexpr size_t kRowSmemMax = 220 * 1024;

// i-columns per tile: shared memory (N1 + 1) BI 16 bytes stays below ~76 KB, so that
// three y CTAs fit on an SM; the widest such tile pads least and keeps a window pass's
// own (sin, cos) in segments of BI 16 bytes (8 columns where 16 fit: 165 us per step
// against 151 at 101^3, 907 against 867 at 200^3).  At the top of a range, edges 288 to
// 297 and 576 to 594, only two z-window CTAs fit, and the wider tile is still no worse:
// per step 2.33 ms with 16 columns and 2.37 with 8 at 288^3, 2.57 both at 290^3, 2.66 and 2.64
// at 293^3; with 8 and 4 columns 18.7 and 20.1 at 576^3, 21.6 and 23.1 at 594^3.
__host__ __device__ inline int cube_tile_lg(int64_t N1) { return N1 <= 297 ? 4 : N1 <= 594 ? 3 : 2; }
__host__ __device__ inline int cube_tile_bi(int64_t N1) { return 1 << cube_tile_lg(N1); }

// Pairs of the cube's x sums ([k][i-block][j][ii]) and of its xy sums
// ([i-block][j][k][ii]): every i-block padded to BI columns.
static int64_t cube_sum_pairs(int64_t N1)
{
    const int BI = cube_tile_bi(N1);
    return ((N1 + BI - 1) / BI) * BI * N1 * N1;
}

static int row_warps(int64_t N1)
{
    const size_t per_warp = (size_t)(N1 + 1) * sizeof(longlong2);
    int w = (int)(kRowSmemMax / per_warp);
    return w < 1 ? 1 : (w > kRowWarpsMax ? kRowWarpsMax : w);
}

// The cube's fused node pass: smaller CTAs than the x pass, so that the shared
// prefix rows of a CTA round up to less of the SM (seven CTAs of four 464-node
// rows, against three of eight).
constexpr int kNodexWarpsMax = 4;
// Shared memory's share of the L1 of the node pass, in percent of its maximum, for rows
// longer than kNodexCarveoutRow<M> nodes.  Left to the driver, long rows take nearly all
// of it for six or seven CTAs per SM and the sin/cos table misses.  Per step in ms, the
// driver's choice and 72%: Kuramoto 3.17 / 3.20 at 320^3, 4.54 / 4.54 at 358^3, 4.73 / 4.72 at
// 362^3, 6.14 / 6.07 at 400^3, 9.99 / 9.48 at 464^3; with inertia 7.37 / 7.52 at 400^3, 9.51 / 9.71
// at 430^3, 11.55 / 11.46 at 464^3, 15.3 / 15.15 at 500^3.  58% and 86% are worse at 464^3.
constexpr int kNodexCarveout = 72;
template <int M> constexpr int64_t kNodexCarveoutRow = M == 0 ? 360 : 448;
// CTAs per SM the fused node pass is compiled for: six for Kuramoto (at most 80
// registers, so stage 4 fits six too), five for the model with inertia.
template <int M> constexpr int kNodexBlocks = M == 0 ? 6 : 5;
static int nodex_warps(int64_t N1)
{
    const int w = row_warps(N1);
    return w > kNodexWarpsMax ? kNodexWarpsMax : w;
}

// The coupled quantity a ball's or disk's window sums add up: the node's (sin,
// cos) on the grid 2^-62 rotated by -alpha = -(rot_q pi/2 + alpha0),
//   e^{-i alpha0} (c + i s) = (c cos a0 + s sin a0) + i (s cos a0 - c sin a0),
// four high products with cos alpha0 and sin alpha0 (non-negative, grid 2^-63),
// which land on the grid 2^-61 (so their truncation leaves no bias that a
// window of millions of terms could accumulate), rounded to nearest onto the
// grid 2^-F, then rot_q quarter turns.  The right-hand side then needs only the
// node's own unrotated (sin, cos) (lattice_coupling).
__device__ __forceinline__ void lattice_rotated_q(const LatticePlan &p, int64_t s62, int64_t c62, int64_t &qs,
                                                  int64_t &qc)
{
    const int sh = 61 - p.F;
    const int64_t h = int64_t(1) << (sh - 1);
    const uint64_t bs = biased62(s62), bc = biased62(c62);
    const int64_t qc4 = (int64_t)(p.rot_c >> 2), qs4 = (int64_t)(p.rot_s >> 2);
    const int64_t c1 = ((int64_t)(__umul64hi(bc, p.rot_c) + __umul64hi(bs, p.rot_s)) + (h - qc4 - qs4)) >> sh;
    const int64_t s1 = ((int64_t)(__umul64hi(bs, p.rot_c) - __umul64hi(bc, p.rot_s)) + (h - qc4 + qs4)) >> sh;
    switch (p.rot_q) { // e^{-i q pi/2}: 1, -i, -1, i
    case 0: qc = c1; qs = s1; break;
    case 1: qc = s1; qs = -c1; break;
    case 2: qc = -c1; qs = -s1; break;
    default: qc = -s1; qs = c1; break;
    }
}

// x pass: one warp per row.  pre[p] = sum_{m<p} Q'(f(m)) for p in [0, N1] is built
// in shared memory as (sin, cos) pairs.  With Pe(p) = pre[p mod N1] + floor(p / N1)
// pre[N1] the periodic extension:
//   MODE 0 (cube)        SX(i) = Pe(i+P+1) - Pe(i-P);
//   MODE 1 (ball, disk,  the extended inclusive prefix E(x) = Pe(x+1),
//           low memory)  x in [-P-1, N1+P-1], modulo 2^64;
//   MODE 2 (ball)        for every half-width w = 0..P the window sums
//                        S_w(i) = Pe(i+w+1) - Pe(i-w), one array of rows per w.
// Modes 1 and 2 build Pe on [-P, N1 + P] (lattice_ext_row) where that fits in shared
// memory; longer rows (disks only, mode 1) extend while they write.
//
// The row's quantities into pre[1..N1] from the stored (sin, cos): the cube's
// unrotated (its node's own phase is turned instead), the ball's and disk's rotated.
template <int MODE>
__device__ __forceinline__ void lattice_row_fill(const LatticePlan &p, int64_t row, longlong2 *pre)
{
    const int lane = threadIdx.x & 31, n1 = (int)p.N1;
    const longlong2 *__restrict__ fr = reinterpret_cast<const longlong2 *>(p.f) + row * n1;
    for (int mb = lane; mb < n1; mb += 32 * 4) { // 4 loads in flight per lane
        longlong2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = mb + 32 * u < n1 ? __ldg(fr + mb + 32 * u) : make_longlong2(0, 0);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (mb + 32 * u < n1) {
                int64_t qs, qc;
                if (MODE == 0) {
                    qs = q62_to(v[u].x, p.F);
                    qc = q62_to(v[u].y, p.F);
                } else lattice_rotated_q(p, v[u].x, v[u].y, qs, qc);
                pre[mb + 32 * u + 1] = make_longlong2(qs, qc);
            }
    }
}

__device__ __forceinline__ longlong2 pair_add(longlong2 a, longlong2 b)
{
    return make_longlong2((long long)((uint64_t)a.x + (uint64_t)b.x), (long long)((uint64_t)a.y + (uint64_t)b.y));
}
__device__ __forceinline__ longlong2 pair_sub(longlong2 a, longlong2 b)
{
    return make_longlong2((long long)((uint64_t)a.x - (uint64_t)b.x), (long long)((uint64_t)a.y - (uint64_t)b.y));
}

// pre[1..n1] -> its inclusive prefix, pre[0] = 0; returns the row's total (wrapping
// sums).  Lanes own an odd number of adjacent slots, so their 16-byte accesses do
// not share banks.
__device__ __forceinline__ longlong2 lattice_row_prefix(longlong2 *pre, int n1)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const int per = ((n1 + 31) >> 5) | 1;
    const int m0 = min(lane * per, n1) + 1, m1 = min(m0 + per, n1 + 1);
    longlong2 r = make_longlong2(0, 0);
    for (int m = m0; m < m1; ++m) r = pair_add(r, pre[m]);
    const longlong2 x = make_longlong2(warp_incl_scan(r.x), warp_incl_scan(r.y));
    longlong2 e = pair_sub(x, r);
    for (int m = m0; m < m1; ++m) {
        e = pair_add(e, pre[m]);
        pre[m] = e;
    }
    if (lane == 0) pre[0] = make_longlong2(0, 0);
    __syncwarp();
    return make_longlong2(__shfl_sync(0xffffffffu, x.x, 31), __shfl_sync(0xffffffffu, x.y, 31));
}

// Window sum at a (0 <= a < n1) of a prefix with its entries `step` pairs apart:
// Pe(a + P + 1) - Pe(a - P).  As 2P + 1 <= n1, at most one end wraps, and either wrap
// adds the total once.
__device__ __forceinline__ longlong2 pair_window(const longlong2 *pre, int n1, int P, int lg, int a, longlong2 total)
{
    const bool wb = a + P + 1 > n1, wl = a < P;
    const int b = a + P + 1 - (wb ? n1 : 0), lo = a - P + (wl ? n1 : 0);
    const longlong2 w = pair_sub(pre[(unsigned)b << lg], pre[(unsigned)lo << lg]);
    return wb || wl ? pair_add(w, total) : w;
}

// The cube's x sums of a row from its prefix, in the plane-wise i-block-major layout
// each y tile reads as one contiguous block: row = k N1 + j; element i at
// ((k tiles + i / BI) N1 + j) BI + i % BI, zeros past the cube's edge.  BI divides 32,
// so a lane's column within its i-block stays fixed and every 32 columns move
// 32 / BI i-blocks further.
__device__ __forceinline__ void cube_x_out(const LatticePlan &p, int64_t row, const longlong2 *pre, longlong2 total)
{
    const int lane = threadIdx.x & 31, n1 = (int)p.N1, P = (int)p.P;
    const int lg = cube_tile_lg(n1), BI = 1 << lg, tiles = (n1 + BI - 1) >> lg;
    const int64_t k = row / n1, j = row - k * n1;
    const unsigned bstep = (unsigned)n1 << lg; // one i-block further
    longlong2 *__restrict__ o = reinterpret_cast<longlong2 *>(p.sx) + ((k * tiles * n1 + j) << lg);
    unsigned at = (unsigned)(lane >> lg) * bstep + (lane & (BI - 1));
#pragma unroll 2
    for (int i = lane; i < tiles << lg; i += 32, at += bstep << (5 - lg))
        o[at] = i < n1 ? pair_window(pre, n1, P, 0, i, total) : make_longlong2(0, 0);
    __syncwarp();
}

// Ball and disk: the row's extended prefix in shared memory, ext[p + P] = Pe(p)
// for p in [-P, N1 + P], then the outputs read straight from it: a window sum is
// two 16-byte shared loads and no wrap test (36 -> 24 us for seven windows of
// 10^6 nodes; the wrapped form took 20 of its 27 instructions per window).
template <int MODE>
__device__ __forceinline__ void lattice_ext_row(const LatticePlan &p, int64_t row, longlong2 *ext)
{
    const int lane = threadIdx.x & 31, n1 = (int)p.N1, P = (int)p.P;
    longlong2 *pre = ext + P; // pre[q] = Pe(q)
    lattice_row_fill<MODE>(p, row, pre);
    const longlong2 total = lattice_row_prefix(pre, n1);
    for (int q = lane; q < P; q += 32) { // 2P + 1 <= N1: both extensions read pre[0..N1]
        pre[q - P] = pair_sub(pre[q - P + n1], total);
        pre[n1 + q + 1] = pair_add(pre[q + 1], total);
    }
    __syncwarp();
    longlong2 *__restrict__ sx = reinterpret_cast<longlong2 *>(p.sx);
    if (MODE == 1) {
        longlong2 *__restrict__ o = sx + row * p.rs;
        for (int e = lane; e < (int)p.rs; e += 32) o[e] = ext[e];
    } else {
        longlong2 *__restrict__ o = sx + row * p.rs;
        const int64_t warray = p.nodes / n1 * p.rs;
        for (int w = 0; w <= P; ++w, o += warray)
#pragma unroll 4
            for (int i = lane; i < n1; i += 32) o[i] = pair_sub(pre[i + w + 1], pre[i - w]);
    }
    __syncwarp();
}

template <int MODE>
__global__ void __launch_bounds__(32 * kRowWarpsMax) lattice_ext_kernel(LatticePlan p)
{
    if (p.skip && *(const volatile int *)p.skip) return;
    extern __shared__ __align__(16) longlong2 ext_mem[];
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int64_t rows = p.nodes / p.N1, row = (int64_t)blockIdx.x * nwarps + warp;
    if (row < rows) lattice_ext_row<MODE>(p, row, ext_mem + warp * (p.N1 + 2 * p.P + 1)); // uniform over the warp
}

// Warps per CTA of lattice_ext_kernel (0: the row's extension does not fit).
static int ext_warps(int64_t N1, int64_t P)
{
    const int64_t w = (int64_t)(kRowSmemMax / (sizeof(longlong2) * (size_t)(N1 + 2 * P + 1)));
    return (int)(w > kRowWarpsMax ? kRowWarpsMax : w);
}

// The x pass of a cube (MODE 0) or of rows too long for lattice_ext_kernel (MODE 1).
template <int MODE>
__global__ void __launch_bounds__(32 * kRowWarpsMax) lattice_x_kernel(LatticePlan p)
{
    if (p.skip && *(const volatile int *)p.skip) return;
    extern __shared__ __align__(16) longlong2 row_mem[];
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5, lane = threadIdx.x & 31;
    const int64_t rows = p.nodes / p.N1, row = (int64_t)blockIdx.x * nwarps + warp;
    if (row >= rows) return; // uniform over the warp
    longlong2 *pre = row_mem + warp * (p.N1 + 1);
    lattice_row_fill<MODE>(p, row, pre);
    const longlong2 total = lattice_row_prefix(pre, (int)p.N1);
    if (MODE == 0) {
        cube_x_out(p, row, pre, total);
    } else { // E(x) = Pe(x + 1) for x in [-P-1, N1+P-1], at slot x + P + 1
        longlong2 *__restrict__ o = reinterpret_cast<longlong2 *>(p.sx) + row * p.rs;
        for (int64_t e = lane; e < p.rs; e += 32) {
            const int64_t q = e - p.P; // = x + 1, in [-P, N1 + P]
            o[e] = q < 0 ? pair_sub(pre[q + p.N1], total) : q > p.N1 ? pair_add(pre[q - p.N1], total) : pre[q];
        }
    }
}

// Deterministic order parameter of the new state: per-CTA partial sums of the
// fixed-point (sin, cos) (exact i128, so the reduction order does not matter),
// and the last CTA to finish sums every partial and records R.  bid / nblk: the
// CTA's index among the network's CTAs of this launch and their number.
// (ps, pc) summed over the CTA, valid in thread 0; every thread of the CTA calls it.
__device__ __forceinline__ void cta_sum_pair(i128 &ps, i128 &pc)
{
    __shared__ i128 s_ws[32], s_wc[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    ps = warp_sum_i128(ps);
    pc = warp_sum_i128(pc);
    __syncthreads(); // an earlier use of s_ws / s_wc is over
    if (lane == 0) {
        s_ws[warp] = ps;
        s_wc[warp] = pc;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        ps = 0;
        pc = 0;
        for (int w = 0; w < nw; ++w) {
            ps += s_ws[w];
            pc += s_wc[w];
        }
    }
}

// The order parameter R = |sum_n e^{i theta_n}| / nodes from the exact sums of
// the n partial pairs at part (p.partial or beyond), by one CTA; recorded in p.obs.
__device__ __forceinline__ void lattice_order_total(const LatticePlan &p, const i128 *part, unsigned n)
{
    i128 ts = 0, tc = 0;
    for (unsigned b = threadIdx.x; b < n; b += blockDim.x) {
        ts += ld_cg_i128(part + 2 * b);
        tc += ld_cg_i128(part + 2 * b + 1);
    }
    cta_sum_pair(ts, tc);
    if (threadIdx.x == 0) {
        const double S = fixed_to_double(ts, p.F), C = fixed_to_double(tc, p.F);
        if (p.obs) {
            const unsigned long long n_rec = *p.obs_ctr;
            p.obs[n_rec % (unsigned long long)p.obs_cap] = sqrt(S * S + C * C) / (double)p.nodes;
            *p.obs_ctr = n_rec + 1;
        }
    }
}

// The CTA's partial sums to p.partial[2 bid, 2 bid + 1]; the last CTA of nblk
// to arrive at *ctr adds them all up and records the order parameter.
__device__ void lattice_record_order(const LatticePlan &p, i128 ps, i128 pc, unsigned bid, unsigned nblk,
                                     unsigned long long *ctr)
{
    __shared__ bool s_last;
    cta_sum_pair(ps, pc);
    if (threadIdx.x == 0) {
        st_i128(p.partial + 2 * bid, ps);
        st_i128(p.partial + 2 * bid + 1, pc);
        __threadfence();
        s_last = last_arrival(ctr, nblk);
    }
    __syncthreads();
    if (!s_last) return;
    lattice_order_total(p, p.partial, nblk);
}

// The order parameter from the partials of a previous launch of nblk CTAs (the
// cube's fused node pass and the ball's and disk's gather, whose CTAs only store
// their partials): CTA g adds up
// its slice of them into the pair nblk + g, and the last of the kOrderCtas CTAs
// to finish (arrival counter tile_ctr) adds those up.
constexpr int kOrderCtas = 128, kOrderThreads = 256;
constexpr unsigned kOrderInline = 1024; // gathers of at most this many CTAs: their last CTA records R itself
                                        // (one launch less; with more CTAs the fences cost more than the launch)
static unsigned order_grid(unsigned nblk) // one CTA per 64 partials, up to kOrderCtas
{
    const unsigned g = (nblk + 63) / 64;
    return g < 1 ? 1u : g > (unsigned)kOrderCtas ? (unsigned)kOrderCtas : g;
}
__global__ void __launch_bounds__(kOrderThreads) lattice_order_kernel(LatticePlan p, unsigned nblk)
{
    if (p.skip && *(const volatile int *)p.skip) return;
    __shared__ bool s_last;
    const unsigned per = (nblk + gridDim.x - 1) / gridDim.x, b0 = blockIdx.x * per, b1 = min(nblk, b0 + per);
    i128 ts = 0, tc = 0;
    for (unsigned b = b0 + threadIdx.x; b < b1; b += blockDim.x) {
        ts += ld_cg_i128(p.partial + 2 * b);
        tc += ld_cg_i128(p.partial + 2 * b + 1);
    }
    cta_sum_pair(ts, tc);
    if (threadIdx.x == 0) {
        st_i128(p.partial + 2 * (nblk + blockIdx.x), ts);
        st_i128(p.partial + 2 * (nblk + blockIdx.x) + 1, tc);
        __threadfence();
        s_last = last_arrival(p.tile_ctr, gridDim.x);
    }
    __syncthreads();
    if (!s_last) return;
    lattice_order_total(p, p.partial + 2 * nblk, gridDim.x);
}

// One node's RK4 stage: right-hand side from the window sums (W0, W1) and its own
// stage input, the RK4 update, the next stage input's local variables and (sin,
// cos).  STAGE 0 (prologue) only computes (sin, cos) of y.  In two parts, so
// that a thread can issue the loads of its next node before it computes this
// one: lattice_node_load reads what the node needs, lattice_node_finish
// computes and writes; lattice_node is the two in a row.
template <int M> struct LatNodeIn {
    int64_t f62[2];                                // (sin, cos) of the stage input, grid 2^-62
    double y[Model<M>::D], acc[Model<M>::D];
    double X[Model<M>::NX > 0 ? Model<M>::NX : 1]; // local stage-input variables
};

template <int M, int STAGE>
__device__ __forceinline__ void lattice_node_load(const LatticePlan &p, int64_t n, LatNodeIn<M> &in)
{
    constexpr int D = Model<M>::D, NX = Model<M>::NX, XOFF = D - NX;
    const int64_t nodes = p.nodes;
#pragma unroll
    for (int v = 0; v < D; ++v) {
        in.y[v] = p.y[v * nodes + n];
        in.acc[v] = STAGE >= 2 ? p.acc[v * nodes + n] : 0.0;
    }
    if (STAGE > 0) {
        const longlong2 v = reinterpret_cast<const longlong2 *>(p.f)[n];
        in.f62[0] = v.x;
        in.f62[1] = v.y;
#pragma unroll
        for (int g = 0; g < NX; ++g) in.X[g] = STAGE == 1 ? in.y[XOFF + g] : p.xs[g * nodes + n];
    }
}

// The RK4 update of a node from its slope k (stages 1-4), the next stage
// input's local variables and (sin, cos); STAGE 0 (prologue) only the (sin,
// cos) of y.  Acc: the type of the thread's order-parameter sums (int64 where a
// thread handles few enough nodes that |sum| <= nodes 2^F stays below 2^63).
template <int M, int STAGE, typename Acc>
__device__ __forceinline__ void lattice_node_update(const LatticePlan &p, int64_t n, const double (&k)[Model<M>::D],
                                                    const LatNodeIn<M> &in, const StepSize &h, bool &ok, Acc &ps,
                                                    Acc &pc, int64_t *sc_out = nullptr)
{
    constexpr int D = Model<M>::D, NX = Model<M>::NX, XOFF = D - NX;
    const int64_t nodes = p.nodes;
    double xn[D];
    if (STAGE == 0) {
#pragma unroll
        for (int v = 0; v < D; ++v) xn[v] = in.y[v];
    } else {
#pragma unroll
        for (int v = 0; v < D; ++v) {
            if (STAGE == 1) {
                p.acc[v * nodes + n] = k[v];
                xn[v] = in.y[v] + h.half * k[v];
            } else if (STAGE == 2) {
                p.acc[v * nodes + n] = in.acc[v] + 2.0 * k[v];
                xn[v] = in.y[v] + h.half * k[v];
            } else if (STAGE == 3) {
                p.acc[v * nodes + n] = in.acc[v] + 2.0 * k[v];
                xn[v] = in.y[v] + h.dt * k[v];
            } else {
                xn[v] = in.y[v] + h.sixth * (in.acc[v] + k[v]);
                p.y[v * nodes + n] = xn[v];
            }
        }
        if (NX > 0 && STAGE <= 3) {
#pragma unroll
            for (int g = 0; g < NX; ++g) p.xs[g * nodes + n] = xn[XOFF + g];
        }
    }
    int64_t s62, c62;
    fixed_sincos(xn[0], p.mp.tab, s62, c62, ok);
    reinterpret_cast<longlong2 *>(p.f)[n] = make_longlong2(s62, c62);
    if (STAGE == 0 || STAGE == 4) {
        ps += q62_to(s62, p.F);
        pc += q62_to(c62, p.F);
    }
    if (sc_out) {
        sc_out[0] = s62;
        sc_out[1] = c62;
    }
}

// The whole node stage: right-hand side from the window sums and the node's own
// stage input, then lattice_node_update.
template <int M, int STAGE, typename Acc>
__device__ __forceinline__ void lattice_node_finish(const LatticePlan &p, int64_t n, int64_t W0, int64_t W1,
                                                    const LatNodeIn<M> &in, const StepSize &h, bool &ok, Acc &ps,
                                                    Acc &pc)
{
    double k[Model<M>::D] = {};
    if (STAGE > 0) Model<M>::rhs_lattice(p.mp, in.f62, W0, W1, in.X, k);
    lattice_node_update<M, STAGE, Acc>(p, n, k, in, h, ok, ps, pc);
}

template <int M, int STAGE>
__device__ __forceinline__ void lattice_node(const LatticePlan &p, int64_t n, int64_t W0, int64_t W1, const StepSize &h,
                                             bool &ok, i128 &ps, i128 &pc)
{
    LatNodeIn<M> in;
    lattice_node_load<M, STAGE>(p, n, in);
    lattice_node_finish<M, STAGE, i128>(p, n, W0, W1, in, h, ok, ps, pc);
}

// ---------------------------------------------------------------------------
// Tiled y and z passes of a cube.  CTA (ib, m) loads the N1 x BI block of pairs of
// one plane (y pass: plane k = m, i-block ib, all j) or one row of columns (z pass:
// row j = m, i-block ib, all k) into shared memory, so that every element crosses
// HBM once.  The block is scanned in place into the exact inclusive prefix along the
// window axis (wrapping int64 arithmetic, as the x pass), and every window sum is
// Pe(a+P+1) - Pe(a-P) on its periodic extension.
constexpr int kTileThreads = 256;

// Asynchronous 16-byte copy global -> shared (both addresses 16-byte aligned).
__device__ __forceinline__ void cp_async16(longlong2 *dst, const longlong2 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__host__ __device__ inline size_t cube_tile_smem(int64_t N1)
{
    return (size_t)(N1 + 1) * (size_t)cube_tile_bi(N1) * sizeof(longlong2);
}

// Load a contiguous block blk[a BI + ii] (a < N1, ii < BI = 2^lg; zeros past the cube's
// edge) into tile[(a + 1) BI + ii] by asynchronous 16-byte copies, so that the whole
// tile is in flight at once, and turn every column into its inclusive prefix along
// a (tile row 0 zero): NT / BI segments per column, the segment sums scanned inside a
// warp by shuffles and across warps from shared memory.  Called by every thread of
// the CTA; ends with a barrier.
template <int NT>
__device__ __forceinline__ void cube_tile_load_scan(const longlong2 *blk, int N1, int lg, longlong2 *tile)
{
    constexpr int NW = NT / 32;
    __shared__ longlong2 s_warp[NW][16];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, BI = 1 << lg;
    for (int e = tid; e < N1 << lg; e += NT) cp_async16(tile + BI + e, blk + e);
    if (tid < BI) tile[tid] = make_longlong2(0, 0);
    cp_async_wait_all();
    __syncthreads();
    const int nseg = NT >> lg, seg = (N1 + nseg - 1) / nseg;
    const int a0 = min((tid >> lg) * seg, N1) + 1, a1 = min(a0 + seg, N1 + 1);
    longlong2 *colp = tile + (tid & (BI - 1));
    longlong2 t = make_longlong2(0, 0);
    for (int a = a0; a < a1; ++a) t = pair_add(t, colp[a << lg]);
    longlong2 x = t; // inclusive over the warp's segments of the column
    for (int d = BI; d < 32; d <<= 1) {
        const longlong2 u = make_longlong2(__shfl_up_sync(0xffffffffu, x.x, d), __shfl_up_sync(0xffffffffu, x.y, d));
        if (lane >= d) x = pair_add(x, u);
    }
    if (lane >= 32 - BI) s_warp[warp][lane & (BI - 1)] = x;
    __syncthreads();
    longlong2 run = pair_sub(x, t);
    for (int w = 0; w < warp; ++w) run = pair_add(run, s_warp[w][lane & (BI - 1)]);
    for (int a = a0; a < a1; ++a) {
        run = pair_add(run, colp[a << lg]);
        colp[a << lg] = run;
    }
    __syncthreads();
}

// Tiled cube y pass: CTA (ib, k); writes the window sums in the i-block-major layout
// the z-window pass reads as one contiguous block (element (ii, j = a, k) at
// ((ib N1 + a) N1 + k) BI + ii; the columns past the cube's edge are zeros already).
// The loop is split where a window wraps, so that most of it tests nothing.
__device__ __forceinline__ void cube_y_tile(const LatticePlan &p, int ib, int k, longlong2 *tile)
{
    const int N1 = (int)p.N1, P = (int)p.P, lg = cube_tile_lg(N1), BI = 1 << lg;
    const int64_t tiles = (N1 + BI - 1) >> lg;
    cube_tile_load_scan<kTileThreads>(reinterpret_cast<const longlong2 *>(p.sx) + ((k * tiles + ib) * N1 << lg), N1, lg, tile);
    const int ii = threadIdx.x & (BI - 1), rstep = kTileThreads >> lg;
    const longlong2 *col = tile + ii;
    const longlong2 total = col[N1 << lg];
    longlong2 *__restrict__ d = reinterpret_cast<longlong2 *>(p.sxy) + (((int64_t)ib * N1 * N1 + k) << lg) + ii;
    const unsigned dstep = (unsigned)N1 << lg;
    int a = threadIdx.x >> lg;
    for (; a < P; a += rstep)
        d[(unsigned)a * dstep] = pair_add(pair_sub(col[(a + P + 1) << lg], col[(a - P + N1) << lg]), total);
#pragma unroll 4
    for (; a < N1 - P; a += rstep) d[(unsigned)a * dstep] = pair_sub(col[(a + P + 1) << lg], col[(a - P) << lg]);
    for (; a < N1; a += rstep)
        d[(unsigned)a * dstep] = pair_add(pair_sub(col[(a + P + 1 - N1) << lg], col[(a - P) << lg]), total);
}

__global__ void __launch_bounds__(kTileThreads) cube_y_tile_kernel(LatticePlan p)
{
    if (p.skip && *(const volatile int *)p.skip) return;
    extern __shared__ __align__(16) longlong2 tile_mem[];
    cube_y_tile(p, blockIdx.x, blockIdx.y, tile_mem);
}

// Batched cubes: CTA b is tile b - yz_base[m] of member m = yz_item[b], in the order of
// the single cube's grid.
__device__ __forceinline__ void cube_batch_tile(const LatticePlan &p, int64_t lb, int &ib, int &m)
{
    const int lg = cube_tile_lg(p.N1), tiles = (int)((p.N1 + (1 << lg) - 1) >> lg);
    m = (int)lb / tiles;
    ib = (int)lb - m * tiles;
}
__global__ void __launch_bounds__(kTileThreads)
    cube_batch_y_kernel(const LatticePlan *__restrict__ plans, const int *__restrict__ yz_item,
                        const int64_t *__restrict__ yz_base)
{
    extern __shared__ __align__(16) longlong2 tile_mem[];
    __shared__ __align__(16) unsigned char plan_mem[sizeof(LatticePlan)];
    LatticePlan &p = *reinterpret_cast<LatticePlan *>(plan_mem);
    const int inst = yz_item[blockIdx.x];
    stage_plan(p, plans + inst);
    int ib, k;
    cube_batch_tile(p, (int64_t)blockIdx.x - yz_base[inst], ib, k);
    cube_y_tile(p, ib, k, tile_mem);
}

// A node's coupling term to cpl (KM = -1), or its whole slope to acc for a
// right-hand-side evaluation of model KM (the stage input's own variables are y).
template <int KM>
__device__ __forceinline__ void lattice_write_slope(const LatticePlan &p, int64_t n, double c)
{
    if constexpr (KM < 0) {
        p.cpl[n] = c;
    } else {
        constexpr int D = Model<KM>::D, NX = Model<KM>::NX, XOFF = D - NX;
        double X[NX > 0 ? NX : 1], k[D];
#pragma unroll
        for (int g = 0; g < NX; ++g) X[g] = p.y[(XOFF + g) * p.nodes + n];
        Model<KM>::rhs_from_coupling(p.mp, c, X, k);
#pragma unroll
        for (int v = 0; v < D; ++v) p.acc[v * p.nodes + n] = k[v];
    }
}

// Ball and disk: from the rotated window sums and the node's own (sin, cos).
template <int KM>
__device__ __forceinline__ void lattice_write_coupling(const LatticePlan &p, int64_t n, int64_t W0, int64_t W1)
{
    const longlong2 f = reinterpret_cast<const longlong2 *>(p.f)[n];
    const int64_t f62[2] = {f.x, f.y};
    lattice_write_slope<KM>(p, n, lattice_coupling_term(p.mp, f62, W0, W1));
}

// Tiled cube z pass, split in two kernels per stage:
//   window pass  CTA (ib, j) scans the xy-window sums of its columns along k and
//                writes every node's coupling term (lattice_coupling_term, the
//                cross product of its own (sin, cos) with its window sums) to
//                cpl; thread (ii, r0) takes the planes k = r0, r0 + kZThreads /
//                BI, ..., the own (sin, cos) of the next two in flight;
//   node pass    one warp per row of consecutive nodes (cube_nodex_kernel): the
//                slope from cpl, the RK4 update, the next (sin, cos), the next
//                stage's x-window sums of the row, and in stage 4 the order
//                parameter's partials.  STAGE 0 is the prologue: the (sin, cos)
//                of y, its x sums and its order parameter.
// The window pass keeps the tile's 64-byte row segments (the z columns are
// N1^2 elements apart), the node pass reads and writes whole warps of
// consecutive nodes.  Three window CTAs per SM up to N1 = 287 and from 298 to 575.
// At 464^3 (interleaved (sin, cos) pairs): two planes per unrolled iteration
// with three planes of prefetch 0.826 ms, two planes of prefetch 0.831 ms, one
// plane per iteration 0.860 ms; 512 threads (at most 42 registers) 0.884 ms.  With
// pairs in the tile too: 0.766 ms.  256 threads and four CTAs per SM take 9.72 ms per
// step against 9.51 at 464^3 (only three fit), 2.70 against 2.77 at 300^3 and 0.859
// against 0.867 at 200^3.
constexpr int kZThreads = 384, kZAhead = 3, kZBlocks = 3; // kZAhead: planes of own (sin, cos) in flight

template <int KM> // -1: coupling terms; a model: the slopes of a right-hand-side evaluation
__device__ __forceinline__ void cube_zw_tile(const LatticePlan &p, int ib, int j, longlong2 *tile)
{
    const int N1 = (int)p.N1, P = (int)p.P, lg = cube_tile_lg(N1), BI = 1 << lg;
    const int i0 = ib << lg, bi = min(BI, N1 - i0);
    const unsigned plane = (unsigned)N1 * (unsigned)N1;
    cube_tile_load_scan<kZThreads>(reinterpret_cast<const longlong2 *>(p.sxy) + (((int64_t)ib * N1 + j) * N1 << lg), N1, lg, tile);
    const int ii = threadIdx.x & (BI - 1), r0 = threadIdx.x >> lg, rstep = kZThreads >> lg;
    if (ii >= bi || r0 >= N1) return; // past every barrier
    const longlong2 *col = tile + ii;
    const longlong2 total = col[N1 << lg];
    const int64_t base = (int64_t)j * N1 + i0 + ii;
    const longlong2 *__restrict__ fp = reinterpret_cast<const longlong2 *>(p.f) + base; // (sin, cos) pairs
    longlong2 f[kZAhead + 1]; // own (sin, cos) of the planes a, a + rstep, ...
#pragma unroll
    for (int d = 0; d < kZAhead; ++d) {
        const int ad = r0 + d * rstep;
        f[d] = ad < N1 ? fp[(unsigned)ad * plane] : make_longlong2(0, 0);
    }
#pragma unroll 2 // two planes' independent chains interleaved
    for (int a = r0; a < N1; a += rstep) {
        const int an = a + kZAhead * rstep;
        f[kZAhead] = an < N1 ? fp[(unsigned)an * plane] : make_longlong2(0, 0);
        const int64_t f62[2] = {f[0].x, f[0].y};
        int64_t t62[2];
        own_phase_turned(p.mp, f62, t62);
        const longlong2 w = pair_window(col, N1, P, lg, a, total);
        lattice_write_slope<KM>(p, base + (unsigned)a * plane, lattice_coupling_term(p.mp, t62, w.x, w.y));
#pragma unroll
        for (int d = 0; d < kZAhead; ++d) f[d] = f[d + 1];
    }
}

template <int KM>
__global__ void __launch_bounds__(kZThreads, kZBlocks) cube_zw_tile_kernel(LatticePlan p)
{
    if (p.skip && *(const volatile int *)p.skip) return;
    extern __shared__ __align__(16) longlong2 tile_mem[];
    cube_zw_tile<KM>(p, blockIdx.x, blockIdx.y, tile_mem);
}

__global__ void __launch_bounds__(kZThreads, kZBlocks)
    cube_batch_zw_kernel(const LatticePlan *__restrict__ plans, const int *__restrict__ yz_item,
                         const int64_t *__restrict__ yz_base)
{
    extern __shared__ __align__(16) longlong2 tile_mem[];
    __shared__ __align__(16) unsigned char plan_mem[sizeof(LatticePlan)];
    LatticePlan &p = *reinterpret_cast<LatticePlan *>(plan_mem);
    const int inst = yz_item[blockIdx.x];
    stage_plan(p, plans + inst);
    int ib, j;
    cube_batch_tile(p, (int64_t)blockIdx.x - yz_base[inst], ib, j);
    cube_zw_tile<-1>(p, ib, j, tile_mem);
}

template <int M, int STAGE>
__device__ __forceinline__ void cube_node_load(const LatticePlan &p, int64_t n, LatNodeIn<M> &in, double &c)
{
    constexpr int D = Model<M>::D, NX = Model<M>::NX, XOFF = D - NX;
    const int64_t nodes = p.nodes;
#pragma unroll
    for (int v = 0; v < D; ++v) {
        in.y[v] = __ldcg(p.y + v * nodes + n); // streamed once: L2 only, L1 left to the sin/cos table
        in.acc[v] = STAGE >= 2 ? __ldcg(p.acc + v * nodes + n) : 0.0;
    }
#pragma unroll
    for (int g = 0; g < NX; ++g) in.X[g] = STAGE <= 1 ? in.y[XOFF + g] : p.xs[g * nodes + n];
    c = STAGE > 0 ? __ldcg(p.cpl + n) : 0.0;
}

// Node pass fused with the next stage's x pass: one warp per row (k, j).  Every
// lane updates its nodes i = lane, lane + 32, ..., and their new (sin, cos)
// rounded onto 2^-F fill the row's prefix rows in shared memory; the row's
// x-window sums then go out in the plane-wise i-block-major layout the y pass
// reads.  In stage 4 (and the prologue, STAGE 0: the (sin, cos) of y, no
// update) the row's sums give the order parameter.
// The loads go through registers, U nodes of a lane ahead: six for Kuramoto
// (compiled for six CTAs per SM, at most 80 registers), four for the model
// with inertia.  Measured on the 464^3 cube, stages 2-4: U = 6 1.18 ms, U = 7 (94
// registers) 1.25 ms, U = 8 1.21 ms, U = 5 (70 registers) 1.34 ms, U = 4
// 1.33 ms; staging the row's y and coupling terms through shared memory by
// cp.async instead took 1.39 ms.  The loads bypass L1 (1% faster).
template <int M, int STAGE>
__device__ __forceinline__ void cube_nodex_row(const LatticePlan &p, const StepSize &h, int64_t row, longlong2 *pre,
                                               bool &ok, int64_t &ps, int64_t &pc)
{
    constexpr int D = Model<M>::D, U = D == 1 ? 6 : 4;
    const int lane = threadIdx.x & 31, n1 = (int)p.N1;
    // the row's own pointers, so that every node address is a 32-bit offset
    const int64_t base = row * p.N1;
    LatticePlan q = p;
    q.y += base;
    q.acc += base;
    q.f += 2 * base; // (sin, cos) pairs
    q.cpl += base;
    if (Model<M>::NX > 0) q.xs += base;
    for (int mb = lane; mb < n1; mb += 32 * U) {
        LatNodeIn<M> in[U];
        double c[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = mb + 32 * u;
            if (i < n1) cube_node_load<M, STAGE>(q, (unsigned)i, in[u], c[u]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = mb + 32 * u;
            if (i < n1) {
                double k[D] = {};
                if (STAGE > 0) Model<M>::rhs_from_coupling(q.mp, c[u], in[u].X, k);
                int64_t sc[2];
                int64_t unused_s = 0, unused_c = 0;
                lattice_node_update<M, STAGE, int64_t>(q, (unsigned)i, k, in[u], h, ok, unused_s, unused_c, sc);
                const int64_t qs = q62_to(sc[0], p.F), qc = q62_to(sc[1], p.F);
                pre[i + 1] = make_longlong2(qs, qc);
                if (STAGE == 0 || STAGE == 4) {
                    ps += qs;
                    pc += qc;
                }
            }
        }
    }
    cube_x_out(p, row, pre, lattice_row_prefix(pre, n1));
}

// CTA bid of a cube's node pass.
template <int M, int STAGE>
__device__ __forceinline__ void cube_nodex_cta(const LatticePlan &p, const StepSize &h, int64_t bid, longlong2 *mem)
{
    const int warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int64_t rows = p.nodes / p.N1, row = bid * nwarps + warp;
    // a lane's order sums: at most ceil(N1 / 32) <= 32 terms of |Q| <= 2^F <= 2^56
    // (F = 61 - ceil(log2 K+) and K+ >= 27), so int64 holds them
    int64_t ps = 0, pc = 0;
    bool ok = true;
    if (row < rows) cube_nodex_row<M, STAGE>(p, h, row, mem + warp * (p.N1 + 1), ok, ps, pc); // uniform over the warp
    if (!ok) raise_error(p.err, ERR_RANGE);
    if (STAGE == 0 || STAGE == 4) { // the order parameter's partials (lattice_order_kernel adds them up)
        i128 ts = ps, tc = pc;
        cta_sum_pair(ts, tc);
        if (threadIdx.x == 0) {
            st_i128(p.partial + 2 * bid, ts);
            st_i128(p.partial + 2 * bid + 1, tc);
        }
    }
}

template <int M, int STAGE>
__global__ void __launch_bounds__(32 * kNodexWarpsMax, kNodexBlocks<M>) cube_nodex_kernel(LatticePlan p, const StepSize h)
{
    extern __shared__ __align__(16) longlong2 row_mem[];
    cube_nodex_cta<M, STAGE>(p, h, blockIdx.x, row_mem);
}

// Batched cubes: CTA b is CTA b - x_base[m] of member m = x_item[b].
template <int M, int STAGE>
__global__ void __launch_bounds__(32 * kNodexWarpsMax, kNodexBlocks<M>)
    cube_batch_nodex_kernel(const LatticePlan *__restrict__ plans, const int *__restrict__ x_item,
                            const int64_t *__restrict__ x_base, const StepSize h)
{
    extern __shared__ __align__(16) longlong2 row_mem[];
    __shared__ __align__(16) unsigned char plan_mem[sizeof(LatticePlan)];
    LatticePlan &p = *reinterpret_cast<LatticePlan *>(plan_mem);
    const int inst = x_item[blockIdx.x];
    stage_plan(p, plans + inst);
    cube_nodex_cta<M, STAGE>(p, h, (int64_t)blockIdx.x - x_base[inst], row_mem);
}

// Order parameters of batched cubes, one CTA per member, from the partials of node
// passes of w rows per CTA.
__global__ void __launch_bounds__(kOrderThreads) cube_batch_order_kernel(const LatticePlan *__restrict__ plans, int w)
{
    const LatticePlan &p = plans[blockIdx.x];
    lattice_order_total(p, p.partial, (unsigned)((p.nodes / p.N1 + w - 1) / w));
}

// ball / disk gather: a thread gathers the window sums of TJ x TK nodes (j,
// j + 1; k, k + 1; disks one plane) at column i.  The plan's table lists the reads
// of all its windows together, (row shift a from row j - P, plane shift z from plane
// k - P, half-width w) in the order of the set of nodes that add them: a row segment
// that several of the windows share is read once (69 reads per node for the 113
// chords of P = 6, 89 with two nodes per thread).  WMODE: one load per read, the
// x-window sum S_w of the row; otherwise two, the difference of the row's
// extended prefix at both ends (wrapping arithmetic; every chord sum and the
// window sum itself are exact either way, so both give the same bits).  Per CTA the
// reads' offsets are put into shared memory with the plane's wrap resolved (two
// reads per 16-byte shared load), so that a read costs a thread the row's wrap, one
// multiply-add and the load.  Rows of window arrays are padded to 8 pairs, and
// threads run over the padded columns, so that 8 lanes read one 128-byte line.
// What bounds it: the L1 data array (16 B per read, and about as much again for the
// lines that arrive from L2).  N1 = 100, P = 6, per stage: one node per thread, with
// both wraps and 64-bit addresses formed per chord, took 36 instructions per chord
// and 152 us; two nodes per thread 88 us; now 84 us.
template <bool WMODE>
__device__ __forceinline__ void gather_read(const longlong2 *base, int j0, int n1, unsigned rowlen, unsigned aw,
                                            unsigned off, uint64_t (&v)[2])
{
    const unsigned jj = (unsigned)j0 + (aw & 0xffffu), jw = min(jj, jj - (unsigned)n1); // row mod N1
    const longlong2 *r = base + (size_t)(off + jw * rowlen);
    if (WMODE) {
        const longlong2 x = __ldg(r);
        v[0] = (uint64_t)x.x;
        v[1] = (uint64_t)x.y;
    } else {
        const int w = (int)(aw >> 16);
        const longlong2 hi = __ldg(r + w), lo = __ldg(r - w - 1);
        v[0] = (uint64_t)hi.x - (uint64_t)lo.x;
        v[1] = (uint64_t)hi.y - (uint64_t)lo.y;
    }
}

// The reads [q, e) of the chunk, which the nodes of the set MASK add.
template <int MASK, int NB, bool WMODE>
__device__ __forceinline__ void gather_class(const uint2 *s_op, int q, int e, const longlong2 *base, int j0, int n1,
                                             unsigned rowlen, uint64_t (&W)[NB][2])
{
    auto add = [&](const uint64_t (&x)[2]) {
#pragma unroll
        for (int b = 0; b < NB; ++b)
            if (MASK >> b & 1) {
                W[b][0] += x[0];
                W[b][1] += x[1];
            }
    };
    if ((q & 1) && q < e) { // to an even read
        const uint2 o = s_op[q++];
        uint64_t x[2];
        gather_read<WMODE>(base, j0, n1, rowlen, o.x, o.y, x);
        add(x);
    }
#pragma unroll (WMODE ? 3 : 2) // measured: 3 reads ahead cost the two-load form registers
    for (; q + 1 < e; q += 2) {
        const uint4 o = *reinterpret_cast<const uint4 *>(s_op + q);
        uint64_t x[2], y[2];
        gather_read<WMODE>(base, j0, n1, rowlen, o.x, o.y, x);
        gather_read<WMODE>(base, j0, n1, rowlen, o.z, o.w, y);
#pragma unroll
        for (int b = 0; b < NB; ++b)
            if (MASK >> b & 1) {
                W[b][0] += x[0] + y[0];
                W[b][1] += x[1] + y[1];
            }
    }
    if (q < e) {
        const uint2 o = s_op[q];
        uint64_t x[2];
        gather_read<WMODE>(base, j0, n1, rowlen, o.x, o.y, x);
        add(x);
    }
}
template <int MASK, int NB, bool WMODE>
__device__ __forceinline__ void gather_classes(const int *start, int c0, int n, const uint2 *s_op,
                                               const longlong2 *base, int j0, int n1, unsigned rowlen,
                                               uint64_t (&W)[NB][2])
{
    if constexpr (MASK < (1 << NB)) {
        const int q = max(start[MASK - 1] - c0, 0), e = min(start[MASK] - c0, n);
        if (q < e) gather_class<MASK, NB, WMODE>(s_op, q, e, base, j0, n1, rowlen, W);
        gather_classes<MASK + 1, NB, WMODE>(start, c0, n, s_op, base, j0, n1, rowlen, W);
    }
}

// STAGE 1-4: the RK4 stage; 0: the prologue (no gather); 5: the slopes into acc (a
// right-hand-side evaluation).  NB nodes per thread (lattice_gather_nodes).
template <int M, int STAGE, bool WMODE, int NB>
__global__ void __launch_bounds__(kGatherThreads, 7) lattice_gather_kernel(LatticePlan p, const StepSize h)
{
    if (STAGE == 5 && p.skip && *(const volatile int *)p.skip) return;
    constexpr int TJ = NB > 1 ? 2 : 1, TK = NB > 2 ? 2 : 1; // rows and planes of a thread's block
    const int n1 = (int)p.N1, P = (int)p.P, tid = threadIdx.x;
    const unsigned cols = (unsigned)(n1 + 7) & ~7u, t = blockIdx.x * kGatherThreads + tid, jp = t / cols;
    const int i = (int)(t - jp * cols), j = TJ * (int)jp, k = TK * blockIdx.y;
    const bool live = i < n1 && j < n1;
    uint64_t W[NB][2] = {};
    if (STAGE > 0) {
        // a read: row shift a | w << 16, and the element offset of its plane (and S_w array)
        __shared__ __align__(16) uint2 s_op[kGatherOps];
        __shared__ int s_start[1 << NB];
        const unsigned rowlen = (unsigned)p.rs;
        const unsigned warray = WMODE ? (unsigned)(p.nodes / n1) * rowlen : 0u; // one S_w
        const bool ball = TK > 1 || p.dims == 3;
        const int j0 = j < P ? j - P + n1 : j - P, k0 = ball ? (k < P ? k - P + n1 : k - P) : 0;
        const longlong2 *base = reinterpret_cast<const longlong2 *>(p.sx) + (live ? i : 0) + (WMODE ? 0 : P + 1);
        const int nops = p.nops;
        if (tid < (1 << NB)) s_start[tid] = p.op_end[tid];
        for (int c0 = 0; c0 < nops; c0 += kGatherOps) {
            const int n = min(kGatherOps, nops - c0);
            if (c0) __syncthreads();
            for (int q = tid; q < n; q += kGatherThreads) {
                const int2 op = __ldg(p.ops + c0 + q); // (a | z << 16, w)
                const int kk = k0 + (op.x >> 16);
                const unsigned kw = ball ? (unsigned)(kk >= n1 ? kk - n1 : kk) : 0u;
                s_op[q] = make_uint2((unsigned)(op.x & 0xffff) | (unsigned)op.y << 16, kw * (unsigned)n1 * rowlen + (unsigned)op.y * warray);
            }
            __syncthreads();
            if (live) gather_classes<1, NB, WMODE>(s_start, c0, n, s_op, base, j0, n1, rowlen, W);
        }
    }
    i128 ps = 0, pc = 0;
    bool ok = true;
    if (live) {
#pragma unroll 1
        for (int kk = 0; kk < TK; ++kk) {
            if (TK > 1 && k + kk >= n1) break;
            const int64_t node = ((int64_t)(k + kk) * n1 + j) * n1 + i;
#pragma unroll
            for (int u = 0; u < TJ; ++u) {
                if (u && j + 1 >= n1) break;
                const int64_t w0 = (int64_t)(kk ? W[NB - TJ + u][0] : W[u][0]), w1 = (int64_t)(kk ? W[NB - TJ + u][1] : W[u][1]);
                if (STAGE == 5) lattice_write_coupling<M>(p, node + u * n1, w0, w1);
                else lattice_node<M, STAGE>(p, node + u * n1, w0, w1, h, ok, ps, pc);
            }
        }
    }
    if (!ok) raise_error(p.err, ERR_RANGE);
    if (STAGE == 0 || STAGE == 4) { // the order parameter's partials
        const unsigned bid = blockIdx.y * gridDim.x + blockIdx.x, nblk = gridDim.x * gridDim.y;
        if (nblk <= kOrderInline) { // the last CTA adds them up
            lattice_record_order(p, ps, pc, bid, nblk, p.done_ctr);
            return;
        }
        cta_sum_pair(ps, pc); // lattice_order_kernel adds them up
        if (tid == 0) {
            st_i128(p.partial + 2 * (int64_t)bid, ps);
            st_i128(p.partial + 2 * (int64_t)bid + 1, pc);
        }
    }
}

// ---------------------------------------------------------------------------
static dim3 tile_grid(int64_t N1)
{
    const int BI = cube_tile_bi(N1);
    return dim3((unsigned)((N1 + BI - 1) / BI), (unsigned)N1, 1);
}

// Nodes per thread of the gather: 4 (rows j, j + 1 of planes k, k + 1) or 2 (rows j,
// j + 1) where the lattice still fills the chip with so few threads.  RK4 step of a
// ball with P = 4, in us, by nodes per thread 4 / 2 / 1: N1 = 40 79 / 59 / 50, 50
// 90 / 71 / -, 64 106 / 97, 72 121 / 173, 100 275 / 327.
int lattice_gather_nodes(int topo, int64_t N1)
{
    if (topo == 3) return N1 >= 400 ? 2 : 1;
    return N1 >= 72 ? 4 : N1 >= 48 ? 2 : 1;
}

// Ball and disk gather: CTAs over (padded column, row or row pair), times planes or
// pairs of them.
static dim3 gather_grid(int topo, int64_t N1)
{
    const int64_t nb = lattice_gather_nodes(topo, N1), tj = nb > 1 ? 2 : 1, tk = nb > 2 ? 2 : 1;
    const int64_t n = (N1 + 7) / 8 * 8 * ((N1 + tj - 1) / tj);
    return dim3((unsigned)((n + kGatherThreads - 1) / kGatherThreads), topo == 3 ? 1u : (unsigned)((N1 + tk - 1) / tk), 1);
}

// Row stride of sx in (sin, cos) pairs: window arrays have rows padded to 8 pairs,
// row prefixes their extension.
int64_t lattice_row_stride(int64_t N1, int64_t P, bool wmode)
{
    return wmode ? (N1 + 7) / 8 * 8 : N1 + 2 * P + 1;
}

int64_t lattice_sx_elems(int topo, int64_t N1, int64_t P, bool wmode)
{
    if (topo == 1) return lattice_sxy_elems(N1);
    const int64_t rows = topo == 3 ? N1 : N1 * N1;
    return 2 * (wmode ? P + 1 : 1) * rows * lattice_row_stride(N1, P, wmode);
}

int64_t lattice_sxy_elems(int64_t N1) { return 2 * cube_sum_pairs(N1); }

int64_t cube_tiles(int64_t N1) { return (N1 + cube_tile_bi(N1) - 1) / cube_tile_bi(N1) * N1; }
int cube_node_warps(int64_t N1) { return nodex_warps(N1); }

int64_t lattice_partial_blocks(int topo, int64_t N1)
{
    // the cube's node pass (one row per warp) or the gather, and the order kernel's second level
    if (topo == 1) return (N1 * N1 + nodex_warps(N1) - 1) / nodex_warps(N1) + kOrderCtas;
    const dim3 g = gather_grid(topo, N1);
    return (int64_t)g.x * g.y + kOrderCtas;
}

cudaError_t lattice_configure()
{
    cudaError_t e = cudaFuncSetAttribute(lattice_x_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kRowSmemMax);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(lattice_x_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)kRowSmemMax);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(lattice_ext_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowSmemMax);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(lattice_ext_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowSmemMax);
    // the largest tile of any edge: the top edge of each tile width
    const int tmax = (int)std::max(std::max(cube_tile_smem(297), cube_tile_smem(594)), cube_tile_smem(1024));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cube_y_tile_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tmax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cube_batch_y_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tmax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cube_batch_zw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, tmax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cube_zw_tile_kernel<-1>, cudaFuncAttributeMaxDynamicSharedMemorySize, tmax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cube_zw_tile_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, tmax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(cube_zw_tile_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, tmax);
#define SIM_NODEX_ATTR(M, S)                                                                                           \
    if (e == cudaSuccess)                                                                                              \
        e = cudaFuncSetAttribute(cube_nodex_kernel<M, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowSmemMax); \
    if (e == cudaSuccess && S > 0)                                                                                     \
        e = cudaFuncSetAttribute(cube_batch_nodex_kernel<M, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowSmemMax);
    SIM_NODEX_ATTR(0, 0) SIM_NODEX_ATTR(0, 1) SIM_NODEX_ATTR(0, 2) SIM_NODEX_ATTR(0, 3) SIM_NODEX_ATTR(0, 4)
    SIM_NODEX_ATTR(3, 0) SIM_NODEX_ATTR(3, 1) SIM_NODEX_ATTR(3, 2) SIM_NODEX_ATTR(3, 3) SIM_NODEX_ATTR(3, 4)
#undef SIM_NODEX_ATTR
    return e;
}

// Batched cube members of one model: the single cube's passes, one launch over all
// members each (every member with its own plan and order-parameter record), so a
// member can be stepped alone or in a batch in any order with the same bits.
// Against sliding windows along j and k (node-order sums, the z pass fused with the
// node update, columns split into segments) a step of 48 networks, rings and cubes
// mixed, took 1.20 ms in place of 1.52.
template <int M>
static cudaError_t cube_batch_stage(int stage, const CubeBatchGroup &g, double dt, cudaStream_t s)
{
    cube_batch_y_kernel<<<(unsigned)g.n_yz, kTileThreads, g.tile_smem, s>>>(g.plans, g.yz_item, g.yz_base);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    cube_batch_zw_kernel<<<(unsigned)g.n_yz, kZThreads, g.tile_smem, s>>>(g.plans, g.yz_item, g.yz_base);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const StepSize h = step_size(dt);
    const unsigned grid = (unsigned)g.n_x, nt = 32u * (unsigned)g.w;
    const size_t smem = sizeof(longlong2) * (size_t)g.w * (size_t)(g.n1_max + 1);
    switch (stage) {
    case 1: cube_batch_nodex_kernel<M, 1><<<grid, nt, smem, s>>>(g.plans, g.x_item, g.x_base, h); break;
    case 2: cube_batch_nodex_kernel<M, 2><<<grid, nt, smem, s>>>(g.plans, g.x_item, g.x_base, h); break;
    case 3: cube_batch_nodex_kernel<M, 3><<<grid, nt, smem, s>>>(g.plans, g.x_item, g.x_base, h); break;
    default:
        cube_batch_nodex_kernel<M, 4><<<grid, nt, smem, s>>>(g.plans, g.x_item, g.x_base, h);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        cube_batch_order_kernel<<<(unsigned)g.n_inst, kOrderThreads, 0, s>>>(g.plans, g.w);
        break;
    }
    return cudaGetLastError();
}

cudaError_t cube_batch_step(const CubeBatchGroup &g, double dt, cudaStream_t s)
{
    if (g.n_x == 0) return cudaSuccess;
    for (int stage = 1; stage <= 4; ++stage) {
        const cudaError_t e = g.model == 3 ? cube_batch_stage<3>(stage, g, dt, s) : cube_batch_stage<0>(stage, g, dt, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

size_t cube_batch_tile_smem(int64_t N1) { return cube_tile_smem(N1); }

// CTAs of a lattice x pass: one row per warp.
static unsigned x_grid(const LatticePlan &p)
{
    const int w = row_warps(p.N1);
    const int64_t rows = p.nodes / p.N1;
    return (unsigned)((rows + w - 1) / w);
}

static size_t x_smem(const LatticePlan &p)
{
    return (size_t)row_warps(p.N1) * (size_t)(p.N1 + 1) * sizeof(longlong2);
}

static cudaError_t launch_x(const LatticePlan &p, cudaStream_t s)
{
    const int w = row_warps(p.N1), we = p.topo == 1 ? 0 : ext_warps(p.N1, p.P);
    if (we > 0) {
        const unsigned grid = (unsigned)((p.nodes / p.N1 + we - 1) / we);
        const size_t smem = sizeof(longlong2) * (size_t)we * (size_t)(p.N1 + 2 * p.P + 1);
        if (p.wmode) lattice_ext_kernel<2><<<grid, 32 * we, smem, s>>>(p);
        else lattice_ext_kernel<1><<<grid, 32 * we, smem, s>>>(p);
    } else if (p.topo == 1) lattice_x_kernel<0><<<x_grid(p), 32 * w, x_smem(p), s>>>(p);
    else lattice_x_kernel<1><<<x_grid(p), 32 * w, x_smem(p), s>>>(p);
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) kernel_mark(s, 0);
    return e;
}

// The cube's y and z-window passes: every node's coupling term (KM = -1) or slope
// of model KM from the x sums.
template <int KM>
static cudaError_t launch_cube_windows(const LatticePlan &p, cudaStream_t s)
{
    cube_y_tile_kernel<<<tile_grid(p.N1), kTileThreads, cube_tile_smem(p.N1), s>>>(p);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    kernel_mark(s, 1);
    cube_zw_tile_kernel<KM><<<tile_grid(p.N1), kZThreads, cube_tile_smem(p.N1), s>>>(p);
    if ((e = cudaGetLastError()) == cudaSuccess) kernel_mark(s, 3);
    return e;
}

// Stage STAGE of a single cube after its x pass: y pass, z-window pass, and the
// node pass fused with the next x pass (STAGE 0: the fused pass alone, the
// prologue).
template <int M, int STAGE>
static cudaError_t launch_cube_stage(const LatticePlan &p, double dt, cudaStream_t s)
{
    cudaError_t e = STAGE > 0 ? launch_cube_windows<-1>(p, s) : cudaSuccess;
    if (e != cudaSuccess) return e;
    const int w = nodex_warps(p.N1);
    const int64_t rows = p.nodes / p.N1;
    const unsigned nblk = (unsigned)((rows + w - 1) / w);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr.val.sharedMemCarveout = kNodexCarveout;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nblk);
    cfg.blockDim = dim3(32 * w);
    cfg.dynamicSmemBytes = (size_t)w * (size_t)(p.N1 + 1) * sizeof(longlong2);
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = p.N1 > kNodexCarveoutRow<M> ? 1 : 0;
    if ((e = cudaLaunchKernelEx(&cfg, cube_nodex_kernel<M, STAGE>, p, step_size(dt))) != cudaSuccess) return e;
    kernel_mark(s, 2);
    if (STAGE == 0 || STAGE == 4) {
        lattice_order_kernel<<<order_grid(nblk), kOrderThreads, 0, s>>>(p, nblk);
        if ((e = cudaGetLastError()) == cudaSuccess) kernel_mark(s, 0);
    }
    return e;
}

template <int M, int STAGE>
static cudaError_t launch_gather(const LatticePlan &p, double dt, cudaStream_t s)
{
    const dim3 grid = gather_grid(p.topo, p.N1);
    const StepSize h = step_size(dt);
    const int nb = lattice_gather_nodes(p.topo, p.N1);
    const bool wm = STAGE > 0 && p.wmode;
    if (nb == 4 && wm) lattice_gather_kernel<M, STAGE, true, 4><<<grid, kGatherThreads, 0, s>>>(p, h);
    else if (nb == 4) lattice_gather_kernel<M, STAGE, false, 4><<<grid, kGatherThreads, 0, s>>>(p, h);
    else if (nb == 2 && wm) lattice_gather_kernel<M, STAGE, true, 2><<<grid, kGatherThreads, 0, s>>>(p, h);
    else if (nb == 2) lattice_gather_kernel<M, STAGE, false, 2><<<grid, kGatherThreads, 0, s>>>(p, h);
    else if (wm) lattice_gather_kernel<M, STAGE, true, 1><<<grid, kGatherThreads, 0, s>>>(p, h);
    else lattice_gather_kernel<M, STAGE, false, 1><<<grid, kGatherThreads, 0, s>>>(p, h);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    kernel_mark(s, 2);
    if ((STAGE == 0 || STAGE == 4) && grid.x * grid.y > kOrderInline) {
        lattice_order_kernel<<<order_grid(grid.x * grid.y), kOrderThreads, 0, s>>>(p, grid.x * grid.y);
        if ((e = cudaGetLastError()) == cudaSuccess) kernel_mark(s, 0);
    }
    return e;
}

// Stage STAGE of a ball or disk: x pass and gather (STAGE 0: the gather alone,
// the prologue).
template <int M, int STAGE>
static cudaError_t launch_gather_stage(const LatticePlan &p, double dt, cudaStream_t s)
{
    const cudaError_t e = STAGE > 0 ? launch_x(p, s) : cudaSuccess;
    return e != cudaSuccess ? e : launch_gather<M, STAGE>(p, dt, s);
}

template <int M>
static cudaError_t launch_stage(int stage, const LatticePlan &p, double dt, cudaStream_t s)
{
    if (p.topo == 1) {
        switch (stage) {
        case 0: return launch_cube_stage<M, 0>(p, dt, s);
        case 1: return launch_cube_stage<M, 1>(p, dt, s);
        case 2: return launch_cube_stage<M, 2>(p, dt, s);
        case 3: return launch_cube_stage<M, 3>(p, dt, s);
        default: return launch_cube_stage<M, 4>(p, dt, s);
        }
    }
    switch (stage) {
    case 0: return launch_gather_stage<M, 0>(p, dt, s);
    case 1: return launch_gather_stage<M, 1>(p, dt, s);
    case 2: return launch_gather_stage<M, 2>(p, dt, s);
    case 3: return launch_gather_stage<M, 3>(p, dt, s);
    default: return launch_gather_stage<M, 4>(p, dt, s);
    }
}

static cudaError_t launch_any(int stage, const LatticePlan &p, double dt, cudaStream_t s)
{
    return p.model == 3 ? launch_stage<3>(stage, p, dt, s) : launch_stage<0>(stage, p, dt, s);
}

// The (sin, cos) of y and its order parameter (the cube: also its x sums).
cudaError_t lattice_prologue(const LatticePlan &p, cudaStream_t s)
{
    return launch_any(0, p, 0.0, s);
}

// k = f(y) into acc, from the stored (sin, cos) of y (y may be a stage input that
// has no x sums yet).
cudaError_t lattice_rhs(const LatticePlan &p, cudaStream_t s)
{
    const cudaError_t e = launch_x(p, s);
    if (e != cudaSuccess) return e;
    if (p.topo == 1) return p.model == 3 ? launch_cube_windows<3>(p, s) : launch_cube_windows<0>(p, s);
    return p.model == 3 ? launch_gather<3, 5>(p, 0.0, s) : launch_gather<0, 5>(p, 0.0, s);
}

cudaError_t lattice_step(const LatticePlan &p, double dt, cudaStream_t s)
{
    for (int stage = 1; stage <= 4; ++stage) {
        const cudaError_t e = launch_any(stage, p, dt, s);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

} // namespace simk
