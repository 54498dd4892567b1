"""The butterfly sum of a block that is not a whole number of warps (hom_warp.h), run on the host:
lanes that the block did not launch hold a value that must not reach the sum, no lane takes from one,
and thread 0 ends with the sum of every thread's value, each once.  Block sizes 1 to 1024."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "hom_warp.h"
// lanes hold powers of two apart by warp, so that a sum names the lanes in it (64-bit counts)
static long long butterfly(long long *v, int n, bool *foreign) {
    for (int off = 16; off > 0; off >>= 1) {
        long long w[32];
        for (int l = 0; l < n; ++l) {
            const bool takes = hom::sum_takes(l, off, n);
            if (takes && (l ^ off) >= n) *foreign = true;
            w[l] = v[l] + (takes ? v[l ^ off] : 0);
        }
        for (int l = 0; l < n; ++l) v[l] = w[l];
    }
    return v[0];
}
int main() {
    for (int threads = 1; threads <= 1024; ++threads) {
        bool foreign = false;
        int lanes = 0;
        for (int w = 0; w < 32; ++w) {
            const int n = hom::warp_lanes(threads, w);
            lanes += n;
            if (n == 0) continue;
            long long v[32];
            for (int l = 0; l < 32; ++l) v[l] = l < n ? 1LL << l : 1LL << 40;   // 2^40: a lane that is not there
            if (butterfly(v, n, &foreign) != (1LL << n) - 1 || foreign) {
                std::printf("%d threads, warp %d\n", threads, w);
                return 1;
            }
        }
        if (lanes != threads) return 2;
    }
    return 0;
}
"""


def test_sum_over_the_lanes_that_exist(tmp_path):
    src, exe = tmp_path / "warp.cpp", tmp_path / "warp"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2110_00733_gb300", "csrc"), str(src), "-o",
                    str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_block_sums_use_it():
    """Every sum over a block of the passes goes through block_sum, and block_sum gives both of its
    warp sums the lanes that the block launched."""
    src = open(os.path.join(ROOT, "paper_2110_00733_gb300", "csrc", "hom_passes.cuh")).read()
    body = src.split("double block_sum(double v) {")[1].split("\n}\n")[0]
    assert body.count("warp_sum(") == body.count("warp_lanes(blockDim.x, ") == 2
