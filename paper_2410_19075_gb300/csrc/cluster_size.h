// CTAs per ring of the cluster-resident kernels (ring_cluster.cu, ring_dp_cluster.cu),
// from the ring and from what the device can co-schedule.
#pragma once
#include <algorithm>
#include <cstdint>

namespace simk {

constexpr int kClusterMaxCtas = 16;
constexpr int kClusterSlice = 512; // RK4: nodes of a CTA at most (|q| < 2^54, so its prefix stays below 2^63)

// RK4 on rings of up to kClusterMaxNodes nodes (HH kClusterMaxNodesHH).  Per step,
// cluster against streaming kernels: KS 10.2 / 21.8 us at N = 5000 and 12.0 / 21.3 us at
// 8192; HH 20.7 / 23.6 us at 5000, 30.5 / 23.1 us at 8192.
constexpr int64_t kClusterMaxNodes = 8192, kClusterMaxNodesHH = 5120;

constexpr int kDpClusterNodes = 8192; // Dormand-Prince: 32 sub-tiles, one lane each in the error sum

// What a device can do: its SMs, and per model the largest cluster it can co-schedule of
// the RK4 and of the Dormand-Prince kernel at their largest slices (0: none, the
// streaming kernels run instead).
struct ClusterLimits {
    int sms = 0;
    int rk4[4] = {0, 0, 0, 0}, dp[4] = {0, 0, 0, 0};
};

// RK4: about 128 nodes per CTA (0: not eligible).
inline int rk4_cluster_size(const ClusterLimits &d, int model, int64_t N)
{
    if (d.rk4[model] < 2 || N > (model == 2 ? kClusterMaxNodesHH : kClusterMaxNodes)) return 0;
    const int cl = (int)std::min<int64_t>(std::max<int64_t>((N + 127) / 128, 2), d.rk4[model]);
    return (N + cl - 1) / cl <= kClusterSlice ? cl : 0;
}

// Dormand-Prince: nodes of a CTA's slice (threads times nodes per thread), and how many of
// them it may fill: a slice's prefix stays below 2^63 in magnitude.  The Kuramoto models'
// |q| reaches 2^53 (a sine or cosine of exactly 1), so 1024 coherent nodes would wrap; the
// others' |q| stays below 2^54 and their slices hold 512.
constexpr int dp_slice(int model) { return model == 0 ? 1024 : model == 2 ? 256 : 512; }
constexpr int dp_slice_nodes(int model) { return model == 0 ? 1023 : dp_slice(model); }

// The fewest CTAs that hold a ring (0: none do, or the device cannot co-schedule them).
inline int dp_cluster_fewest(const ClusterLimits &d, int model, int64_t N)
{
    if (N > kDpClusterNodes) return 0;
    for (int cl = 1; cl <= d.dp[model]; ++cl) {
        const int64_t per = ((N + cl - 1) / cl + 31) / 32 * 32; // the kernel's slices, all but the last one full
        if (per <= dp_slice(model) && std::min(per, N) <= dp_slice_nodes(model)) return cl;
    }
    return 0;
}

// A run whose rings at their fewest CTAs fill the chip (two CTAs per SM) more than twice
// over is bound by throughput, not by its longest chain.  There the streaming kernels are
// the faster ones for Hodgkin-Huxley rings of more than 1024 nodes and FitzHugh-Nagumo
// rings of more than 2560 (256 rings, streaming against cluster: HH 38.3 / 38.3 ms at 1100
// nodes, 45.4 / 48.7 at 1500, 82.6 / 97.0 at 3000; FHN 31.5 / 30.0 at 2100, 42.4 / 43.8 at
// 3000, 58.2 / 61.3 at 4100); the Kuramoto models gain at every size (4.07 / 3.30 at 4100).
inline bool dp_run_is_full(const ClusterLimits &d, int64_t fewest_ctas) { return fewest_ctas > 4 * (int64_t)d.sms; }
constexpr int64_t dp_full_run_nodes(int model) { return model == 2 ? 1024 : model == 1 ? 2560 : kDpClusterNodes; }

// CTAs per ring of a run of n_rings rings (full: dp_run_is_full): the fewest that hold the
// ring, or more, a power of two, while the rings still fit on the chip together and a CTA
// keeps at least 96 nodes.  0: dp_launch's kernels.
inline int dp_cluster_size(const ClusterLimits &d, int model, int64_t N, int n_rings, bool full = false)
{
    int cl = dp_cluster_fewest(d, model, N);
    if (cl == 0 || (full && N > dp_full_run_nodes(model))) return 0;
    for (int c = 2; c <= d.dp[model]; c *= 2)
        if (c > cl && (int64_t)n_rings * c <= 2 * d.sms && N / c >= 96) cl = c;
    return cl;
}

// One of few cluster sizes for a ring of cl CTAs: the next power of two, if the device takes it.
inline int dp_cluster_class(const ClusterLimits &d, int model, int cl)
{
    int c = 1;
    while (c < cl) c *= 2;
    return c <= d.dp[model] ? c : cl;
}

} // namespace simk
