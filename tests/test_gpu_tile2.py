"""Every accepted explicit tile2 runs: a tile of one column, 8 bytes wide, is no TMA copy (those start and
end on 16-byte boundaries) and takes the plain-load n2 pass.  Against numpy's DFT; an FP32 transform of two
or three stages an axis carries a few eps = 6e-8 per stage, 5e-6 leaves an order of magnitude."""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile2", [1, 2, 4])
@pytest.mark.parametrize("n", [16, 45, 48, 64, 108, 256])
def test_narrow_tiles_are_the_dft(n, tile2):
    from paper_2110_00733_gb300 import build, hom
    build.build()
    hom.load_library()
    g = (3, n, 10)
    f = ri.random_field(g, 7).astype(np.float32)
    ref = np.moveaxis(np.fft.rfftn(f.astype(np.float64), axes=(1, 2, 3)), 0, -1)
    with hom.hom_create(g, np.ones(g, dtype=np.float32), shape=(0, tile2, 0)) as ctx:
        s = hom.hom_fft_forward(ctx, f)
        assert np.linalg.norm(s - ref) <= 5e-6 * np.linalg.norm(ref)
        assert np.linalg.norm(hom.hom_fft_inverse(ctx, s) - f) <= 5e-6 * np.linalg.norm(f)
