"""The three-float sum of products (hom_sum3.h), run on the host against 128-bit arithmetic: squares, whose
last bits are not random, and products of both signs, 1 to 4096 of them, over ten decades.  The leading two
floats are exact, the third rounds at 2^-24 of what they leave (2^-46 of the sum): n such roundings are
below n 2^-70, and value() rounds once to FP64 (2^-53).  For products of both signs the same of the sum of
their absolute values."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdint>
#include <cstdio>
#include <cmath>
#include "hom_sum3.h"
static uint64_t s = 88172645463325252ull;
static double uni() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return (double)(s >> 11) * 0x1p-53; }
int main() {
    for (int kind = 0; kind < 3; ++kind)
        for (int n = 1; n <= 4096; n *= 2)
            for (int rep = 0; rep < 200; ++rep) {
                hom::Sum3 t;
                long double ex = 0, exl = 0, mag = 0;   // exact sum in two parts (products have 48 bits)
                for (int i = 0; i < n; ++i) {
                    const float a = (float)((2 * uni() - 1) * std::pow(10.0, kind == 2 ? -10 * uni() : -uni()));
                    const float b = kind == 0 ? a : (kind == 2 ? 2 * a : (float)(2 * uni() - 1));
                    t.add_prod(a, b);
                    const long double p = (long double)a * b, q = ex + p, bb = q - ex;
                    exl += (ex - (q - bb)) + (p - bb);
                    ex = q;
                    mag += p < 0 ? -p : p;
                }
                const long double err = ((long double)t.value() - ex) - exl;
                if (std::fabs(err) > (0x1p-53L + n * 0x1p-70L) * mag * 1.01L) {
                    std::printf("kind %d n %d: %Lg of %Lg\n", kind, n, err, mag);
                    return 1;
                }
            }
    return 0;
}
"""


def test_as_good_as_64_bits(tmp_path):
    src, exe = tmp_path / "sum3.cpp", tmp_path / "sum3"
    src.write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2110_00733_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
