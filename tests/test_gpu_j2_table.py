"""An elastoplastic increment with its projector's unit vectors formed in the passes, as where their table
cannot be allocated, against the same increment with the table: the same operations, so the same bits."""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("deriv", ["rotated", "continuous"])
@pytest.mark.parametrize("g", [(16, 16, 16), (18, 20, 24), (25, 32, 27)])
def test_increment_without_the_table(monkeypatch, g, deriv):
    from paper_2110_00733_gb300 import build, hom
    build.build()
    hom.load_library()
    phi = np.ascontiguousarray(ri.random_phi(g, 23), dtype=np.float64)
    d = hom.HOM_DERIV_ROTATED if deriv == "rotated" else hom.HOM_DERIV_CONTINUOUS
    out, size = [], []
    for table in ("1", "0"):
        monkeypatch.setenv("HOM_J2_TABLE", table)
        with hom.hom_create(g, phi, hom.HOM_INPUT_FRACTION_F64, 1.0e9, 0.3, precision=hom.HOM_PREC_FP64, derivative=d) as c:
            hom.hom_j2_begin(c, 2.0e7, 0.0)
            hom.hom_j2_increment(c, [-0.03, 0, 0, 0, 0, 0], np.zeros(6), 0b000110, max_newton=2, max_lin=25)
            out.append(hom.hom_j2_state(c))
            size.append(hom.hom_get_info(c)[2])
    assert size[0] - size[1] == 48 * g[0] * g[1] * (g[2] // 2 + 1)   # one has the table, the other has not
    for a, b in zip(*out):
        assert np.array_equal(a, b) and np.abs(a).max() > 0
