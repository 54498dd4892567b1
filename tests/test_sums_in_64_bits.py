"""Which sums of the persistent FP32 passes run in FP64, by reading their source (an error of 1e-13 in a
norm is far below what an FP32 field shows): ||u_{k+1}||^2 over a CTA's tiles and the strain energies over
its rows.  Two floats over all tiles of a case drift with their number, one tile's products do not; the
emulation below gives both figures."""
import os

import numpy as np

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_00733_gb300", "csrc")


def kernel(name, fn):
    """The body of a __global__ function, from its name to the closing brace in column one."""
    src = open(os.path.join(CSRC, fn)).read()
    at = src.index(name + "(Geometry g")
    return src[at:src.index("\n}\n", at)]


def test_norm_over_tiles():
    body = kernel("k_x1_lanczos_tma", "hom_lines.cuh")
    assert "double run = 0.0;" in body and "run += acc.value();" in body
    loop = body[body.index("for (int i = 0; tile < ntiles; ++i)"):]
    assert "Acc<R> acc;" in loop and "Acc<R> acc;" not in body[:body.index("for (int i = 0; tile < ntiles; ++i)")]


def test_energies_over_rows():
    for name, fn in (("k_x3_line", "hom_x3.cuh"), ("k_x3r", "hom_passes.cuh")):
        body = kernel(name, fn)
        assert "double eacc = 0.0;" in body and "eacc += (double)en;" in body, name


def test_two_floats_drift_over_tiles():
    f4, f8 = np.float32, np.float64
    rng = np.random.default_rng(2)
    threads, tiles, per = 2048, 36, 16   # 256^3: products of a thread in one tile, tiles of a CTA
    hi, lo = np.zeros(threads, f4), np.zeros(threads, f4)
    run, exact = np.zeros(threads), np.zeros(threads, np.longdouble)

    def add(h, low, q):
        p = (q.astype(f8) * q).astype(f4)
        e = (q.astype(f8) * q - p).astype(f4)
        s = h + p
        b = s - h
        return s, low + (((h - (s - b)) + (p - b)) + e)

    for _ in range(tiles):
        th, tl = np.zeros(threads, f4), np.zeros(threads, f4)
        for _ in range(per):
            q = rng.standard_normal(threads).astype(f4)
            hi, lo = add(hi, lo, q)
            th, tl = add(th, tl, q)
            exact += q.astype(np.longdouble) ** 2
        run += th.astype(f8) + tl
    rms = lambda v: float(np.sqrt(np.mean(((v - exact) / exact).astype(f8) ** 2)))  # noqa: E731
    assert rms(run) < 5e-15 < 5e-14 < rms(hi.astype(f8) + lo)
