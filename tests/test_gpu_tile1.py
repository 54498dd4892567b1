"""An explicit tile1 is the unfused n1 passes' tile; the fused MINRES pass stays the TMA-staged one of its
own tile.  No value depends on the tile it is computed in, so a few steps return the same bits as with the
automatic shape (the plain-load fused pass, which rounds in another order, does not)."""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n, tile1", [(160, 4), (160, 1), (96, 2), (108, 1), (256, 1), (18, 8), (240, 3)])
def test_fused_pass_keeps_its_tile(n, tile1):
    from paper_2110_00733_gb300 import build, hom
    build.build()
    hom.load_library()
    g = (n, 5, 12)
    phi = ri.random_phi(g, 17)
    E = np.array([[1e-3, 2e-4, -3e-4, 1e-4, 3e-4, -2e-4], [0, 0, 1e-3, 0, 0, 5e-4]])
    got = []
    for shape in ((0, 0, 0), (0, 0, tile1)):
        with hom.hom_create(g, phi, hom.HOM_INPUT_FRACTION_F64, shape=shape, refine=0) as ctx:
            rc, info = hom.hom_solve(ctx, E, tol=1e-12, max_it=7)
            assert rc == hom.HOM_NOT_CONVERGED and [i["iterations"] for i in info] == [7, 7]
            got.append([hom.hom_fields(ctx, k, want=("stress",))[1] for k in range(2)])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
