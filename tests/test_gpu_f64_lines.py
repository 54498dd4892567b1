"""FP64 passes on the line engine at every length it takes, on each axis.

Tolerances.  An FP64 transform with 2 or 3 stages per axis carries a relative
error of a few eps = 1.1e-16 per stage; the operator transforms there and back
and projects twice: 1e-13 of the result's norm leaves an order of magnitude.
Seven MINRES steps in FP64 and FP32 from the same right-hand side differ by the
FP32 ones' rounding: 5e-6 of the stress field's norm.
"""
import numpy as np
import pytest

import oracle
import rve_inputs as ri

pytestmark = pytest.mark.gpu

LENGTHS = [8] + sorted(2 ** a * 3 ** b * 5 ** c for a in range(10) for b in range(6) for c in range(4)
                       if 16 <= 2 ** a * 3 ** b * 5 ** c <= 512)


@pytest.fixture(scope="module")
def hom():
    from paper_2110_00733_gb300 import build
    build.build()
    from paper_2110_00733_gb300 import hom as h
    h.load_library()
    return h


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", LENGTHS)
def test_f64_operator_and_solve(hom, n, axis):
    g = [3, 5, 6]
    g[axis] = n
    g = tuple(g)
    phi = ri.random_phi(g, 17)
    half = lambda x: np.ascontiguousarray(np.moveaxis(np.fft.rfftn(x, axes=(1, 2, 3)), 0, -1))
    f = ri.random_field(g, 19)
    spec, ref = half(f), half(oracle.apply(phi, 1.0, 0.3, 1, oracle.project(g, 1, f)))
    E = np.array([[1e-3, 2e-4, -3e-4, 1e-4, 3e-4, -2e-4]])
    sig = []
    for prec in (hom.HOM_PREC_FP64, hom.HOM_PREC_FP32_FIELDS):
        with hom.hom_create(g, phi, hom.HOM_INPUT_FRACTION_F64, precision=prec) as ctx:
            if prec == hom.HOM_PREC_FP64:
                got = hom.hom_apply_spectrum(ctx, spec)
                assert np.linalg.norm(got - ref) <= 1e-13 * np.linalg.norm(ref)
            _, info = hom.hom_solve(ctx, E, tol=1e-12, max_it=7)
            assert info[0]["iterations"] == 7
            sig.append(hom.hom_fields(ctx, 0, want=("stress",))[1])
    assert np.linalg.norm(sig[0] - sig[1]) <= 5e-6 * np.linalg.norm(sig[0])
