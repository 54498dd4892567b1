"""MoDBFFT conjugate gradients on loads of very different size (section 2.2)."""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hom():
    import torch
    assert torch.cuda.is_available()
    from paper_2110_00733_gb300 import build, hom as h
    build.build()
    h.load_library()
    return h


@pytest.mark.parametrize("shape", [(18, 20, 24), (9, 15, 25), (64, 64, 12)])
def test_pcg_scales_with_the_load(hom, shape):
    """A load scaled by a power of two gives the same iterates, scaled: the sums of the FP32 step
    are taken of products brought into the range of FP32 by a power of two.  Everything is exact
    under that scaling but the smallest products' last bits (far below 1e-9 of the sums)."""
    phi = ri.random_phi(shape, seed=5, void_fraction=0.3)
    out = []
    for s in (1.0, 2.0 ** -45):
        with hom.hom_create(shape, np.ascontiguousarray(phi, dtype=np.float64), hom.HOM_INPUT_FRACTION_F64, 110e9, 0.3,
                            derivative=hom.HOM_DERIV_CONTINUOUS, solver=hom.HOM_SOLVER_MODBFFT_CG) as c:
            _, info = hom.hom_solve(c, [0.01 * s, 0.0, 0.0, 0.002 * s, 0.0, 0.0], tol=1e-7, max_it=12)
            out.append((np.asarray(info[0]["sigma_mean"]) / s, info[0]["iterations"]))
    assert out[0][1] == out[1][1] and out[0][1] > 2
    np.testing.assert_allclose(out[1][0], out[0][0], rtol=1e-9, atol=1e-9 * np.abs(out[0][0]).max())
