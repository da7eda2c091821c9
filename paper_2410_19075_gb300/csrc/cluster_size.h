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

// CTAs per ring of a run of n_rings rings: as few as hold the ring when the rings alone
// fill the chip (two CTAs per SM), more while they do not and a CTA keeps at least 96
// nodes.  0: dp_launch's kernels.
inline int dp_cluster_size(const ClusterLimits &d, int model, int64_t N, int n_rings)
{
    const int maxc = d.dp[model];
    if (N > kDpClusterNodes) return 0;
    auto fits = [&](int cl) {
        const int64_t per = ((N + cl - 1) / cl + 31) / 32 * 32; // the kernel's slices, all but the last one full
        return per <= dp_slice(model) && std::min(per, N) <= dp_slice_nodes(model);
    };
    int cl = 1;
    while (cl <= maxc && !fits(cl)) cl *= 2;
    if (cl > maxc) return 0;
    while (cl * 2 <= maxc && (int64_t)n_rings * cl * 2 <= 2 * d.sms && N / (2 * cl) >= 96) cl *= 2;
    return cl;
}

} // namespace simk
