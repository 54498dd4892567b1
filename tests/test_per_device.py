"""Values made once per device (per_device.h), run on the host: each device has its own, made once
whatever the number of threads; one that could not be made is tried again; no device, no value."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <atomic>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
    hnet::PerDevice<int> p;
    std::atomic<int> made{0}, wrong{0};
    auto work = [&] {
        for (int k = 0; k < 2000; ++k) {
            const int dev = k % 8;
            int *v = p.get(dev, [&](int &x) { ++made; x = 100 + dev; return true; });
            if (!v || *v != 100 + dev) ++wrong;
        }
    };
    std::vector<std::thread> t;
    for (int i = 0; i < 8; ++i) t.emplace_back(work);
    for (auto &x : t) x.join();
    if (made != 8 || wrong) return 1;
    auto ok = [](int &x) { x = 7; return true; };
    auto fails = [](int &x) { x = 9; return false; };
    if (p.get(0, ok) == p.get(1, ok)) return 2;                                   // one each
    if (p.get(20, fails) || !p.get(20, ok) || *p.get(20, fails) != 7) return 3;   // tried again, then kept
    return p.get(-1, ok) || p.get(64, ok) ? 4 : 0;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "pd.cpp", tmp_path / "pd"
    src.write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", os.path.join(ROOT, "paper_2110_00733_gb300", "csrc"), str(src),
                    "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_network_launchers_keep_no_other_static():
    """What the launchers keep between calls is made per device and under a lock: kernel attributes and
    the number of SMs belong to a device, and a plain flag is written by every thread that finds it unset."""
    import re
    for name in ("net.cu", "net_tc.cu"):
        src = open(os.path.join(ROOT, "paper_2110_00733_gb300", "csrc", name)).read()
        kept = re.findall(r"^\s+static (?!constexpr)([^;(]*)", src, re.M)
        assert all(k.startswith(("PerDevice<", "const int regs")) for k in kept), kept
