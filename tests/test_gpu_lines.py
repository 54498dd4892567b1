"""The line engine's passes (TMA-staged n2 pass, fused MINRES n1 pass) at every
length they take, against numpy's DFT and against the plain-load passes.

Tolerances.  An FP32 transform of length N with 2 or 3 stages per axis carries
a relative L2 error of a few eps = 6e-8 per stage: 5e-6 of the result's norm
leaves an order of magnitude.  Seven MINRES iterations from the same
right-hand side differ between two FP32 evaluations by their rounding, a few
eps each, not amplified over so few steps: 5e-6 of the stress field's norm.
"""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu

LENGTHS = sorted(2 ** a * 3 ** b * 5 ** c for a in range(10) for b in range(6) for c in range(4)
                 if 16 <= 2 ** a * 3 ** b * 5 ** c <= 512)


@pytest.fixture(scope="module")
def hom():
    from paper_2110_00733_gb300 import build
    build.build()
    from paper_2110_00733_gb300 import hom as h
    h.load_library()
    return h


@pytest.mark.parametrize("n", LENGTHS)
def test_n2_pass_is_the_dft(hom, n):
    g = (3, n, 10)
    f = ri.random_field(g, 7).astype(np.float32)
    ref = np.moveaxis(np.fft.rfftn(f.astype(np.float64), axes=(1, 2, 3)), 0, -1)
    phi = np.ones(g, dtype=np.float32)
    with hom.hom_create(g, phi) as ctx:
        s = hom.hom_fft_forward(ctx, f)
        assert np.linalg.norm(s - ref) <= 5e-6 * np.linalg.norm(ref)
        back = hom.hom_fft_inverse(ctx, s)
        assert np.linalg.norm(back - f) <= 5e-6 * np.linalg.norm(f)


@pytest.mark.parametrize("n", LENGTHS)
def test_fused_n1_pass_matches_plain_loads(hom, n):
    g = (n, 5, 12)   # 35 columns: ragged last tile for most tile widths
    phi = ri.random_phi(g, 11)
    E = np.array([[1e-3, 2e-4, -3e-4, 1e-4, 3e-4, -2e-4], [0, 0, 1e-3, 0, 0, 5e-4]])
    got = []
    for staging in (0, 1):
        with hom.hom_create(g, phi, hom.HOM_INPUT_FRACTION_F64, staging=staging) as ctx:
            rc, info = hom.hom_solve(ctx, E, tol=1e-12, max_it=7)
            assert rc == hom.HOM_NOT_CONVERGED and [i["iterations"] for i in info] == [7, 7]
            got.append([hom.hom_fields(ctx, k, want=("stress",))[1] for k in range(2)])
    for a, b in zip(*got):
        assert np.linalg.norm(a - b) <= 5e-6 * np.linalg.norm(b)


@pytest.mark.parametrize("n", LENGTHS)
def test_n3_pass_matches_the_shared_memory_pass(hom, n):
    """The persistent n3 pass (law and strain energy) against the pass that an
    explicit rows3 selects: the operator, and a solve, whose alpha is the
    pass's energy.  45 rows: ragged last tile."""
    g = (5, 9, n)
    phi = ri.random_phi(g, 13)
    E = np.array([[1e-3, 2e-4, -3e-4, 1e-4, 3e-4, -2e-4], [0, 0, 1e-3, 0, 0, 5e-4]])
    spec = np.fft.rfftn(ri.random_field(g, 5), axes=(1, 2, 3))
    spec = np.ascontiguousarray(np.moveaxis(spec, 0, -1)).astype(np.complex64)
    got = []
    for rows in (0, 2):
        with hom.hom_create(g, phi, hom.HOM_INPUT_FRACTION_F64, shape=(rows, 0, 0)) as ctx:
            out = [hom.hom_apply_spectrum(ctx, spec)]
            rc, info = hom.hom_solve(ctx, E, tol=1e-12, max_it=7)
            assert rc == hom.HOM_NOT_CONVERGED and [i["iterations"] for i in info] == [7, 7]
            got.append(out + [hom.hom_fields(ctx, k, want=("stress",))[1] for k in range(2)])
    for a, b in zip(*got):
        assert np.linalg.norm(a - b) <= 5e-6 * np.linalg.norm(b)
