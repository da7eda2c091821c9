"""CTAs per ring of the cluster-resident kernels, from what a device can co-schedule."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2410_19075_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include "cluster_size.h"

// args: sms, largest RK4 cluster, largest Dormand-Prince cluster; reads lines "model N rings"
int main(int, char **v)
{
    simk::ClusterLimits d;
    d.sms = std::atoi(v[1]);
    for (int m = 0; m < 4; ++m) d.rk4[m] = std::atoi(v[2]), d.dp[m] = std::atoi(v[3]);
    int model, rings;
    long long n;
    while (std::scanf("%d %lld %d", &model, &n, &rings) == 3) {
        const int cl = simk::dp_cluster_size(d, model, n, rings), full = simk::dp_cluster_size(d, model, n, rings, true);
        std::printf("%d %d %d %d %d %d\n", simk::rk4_cluster_size(d, model, n), cl, simk::dp_slice(model),
                    simk::dp_slice_nodes(model), full, cl ? simk::dp_cluster_class(d, model, cl) : 0);
    }
}
"""

MAX_Q = {0: 2 ** 53, 1: 2 ** 54 - 1, 2: 2 ** 54 - 1, 3: 2 ** 53}  # largest coupled quantity on its grid


@pytest.fixture(scope="module")
def sizes(tmp_path_factory):
    d = tmp_path_factory.mktemp("cluster_size")
    (d / "main.cpp").write_text(MAIN)
    exe = str(d / "main")
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, str(d / "main.cpp"), "-o", exe], check=True)

    def run(sms, rk4, dp, rings):
        text = "".join(f"{m} {n} {k}\n" for m, n, k in rings)
        out = subprocess.run([exe, str(sms), str(rk4), str(dp)], input=text, check=True, capture_output=True, text=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    return run


NODES = sorted({*range(2, 70), 255, 256, 257, *range(990, 1060), 2047, 2048, 2049, 4064, 4095, 4096, 4097, 5119, 5120, 5121,
                *range(7930, 7945), 8191, 8192, 8193, 10 ** 6})


@pytest.mark.parametrize("largest", [0, 1, 2, 4, 8, 16])
@pytest.mark.parametrize("sms", [1, 132, 148, 152])
def test_slices_fit_and_do_not_wrap(sizes, sms, largest):
    rings = [(m, n, k) for m in range(4) for n in NODES for k in (1, 24, 200, 1000)]
    for (m, n, k), (rk4, dp, slots, filled, full, cls) in zip(rings, sizes(sms, largest, largest, rings)):
        # no kernel whose own shape the device cannot co-schedule: 0 is the streaming kernels
        assert 0 <= rk4 <= largest and 0 <= dp <= cls <= largest
        assert filled * MAX_Q[m] < 2 ** 63 and 512 * MAX_Q[m] < 2 ** 63
        if rk4:
            assert n <= (5120 if m == 2 else 8192) and -(-n // rk4) <= 512

        def per(c):  # nodes of a slice, and slots
            slice_slots = -(-(-(-n // c)) // 32) * 32
            return slice_slots <= slots and min(slice_slots, n) <= filled
        fewest = next((c for c in range(1, largest + 1) if n <= 8192 and per(c)), 0)
        assert (dp > 0) == (fewest > 0) and full in (0, dp)
        if dp:
            assert per(dp) and per(cls)
            # more than the fewest only while the chip is not full
            assert dp == fewest or (dp > fewest and k * dp <= 2 * sms and n // dp >= 96)
            assert (full == 0) == (n > {0: 8192, 1: 2560, 2: 1024, 3: 8192}[m])


def test_the_two_kernels_are_asked_separately(sizes):
    """A device that takes 16 small RK4 CTAs, but only 4 of the Dormand-Prince kernel's 106 KB
    (4000 nodes in four would fill slices of 1024)."""
    rings = [(0, 4000, 1), (0, 8192, 1), (2, 1024, 1), (2, 1025, 1)]
    assert [r[:2] for r in sizes(152, 16, 4, rings)] == [(16, 0), (16, 0), (8, 4), (9, 0)]
    assert [r[:2] for r in sizes(152, 0, 0, rings)] == [(0, 0)] * 4
