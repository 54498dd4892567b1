"""The FP64 passes of an elastoplastic increment on compile-time plans (ordered_fft, narrow tiles)
against the runtime engine, which explicit launch shapes select: the same operations in the same
order, so the same bits, although an increment amplifies rounding a billionfold."""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hom():
    from paper_2110_00733_gb300 import build
    build.build()
    from paper_2110_00733_gb300 import hom as h
    h.load_library()
    return h


# n1 of at most 32 and not a register length: the runtime engine's tile1 is 16 there
@pytest.mark.parametrize("g", [(18, 20, 24), (24, 45, 50), (30, 27, 54), (20, 81, 25), (25, 32, 60), (27, 40, 125)])
def test_increment_repeats_the_runtime_engine(hom, g):
    phi = np.ascontiguousarray(ri.random_phi(g, 21), dtype=np.float64)
    out = []
    for shape in ((0, 0, 0), (3, 8, 16)):
        with hom.hom_create(g, phi, hom.HOM_INPUT_FRACTION_F64, 1.0e9, 0.3, precision=hom.HOM_PREC_FP64, shape=shape) as c:
            hom.hom_j2_begin(c, 2.0e7, 0.0)
            hom.hom_j2_increment(c, [-0.03, 0, 0, 0, 0, 0], np.zeros(6), 0b000110, max_newton=2, max_lin=25)
            out.append(hom.hom_j2_state(c))
    for a, b in zip(*out):
        assert np.array_equal(a, b) and np.abs(a).max() > 0
