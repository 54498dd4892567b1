"""The FP64 n2 pass at every width its tiles take: 32 columns (odd threads a line), 16 and 8 (9 and 10 threads,
with many columns and with few), and the runtime engine at 384, against numpy's DFT.  An FP64 transform of two
or three stages carries a few times 1e-16: 1e-14 of the result's norm leaves an order of magnitude."""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("g", [(3, 25, 10), (40, 25, 60), (64, 75, 64), (3, 90, 10), (40, 90, 60), (8, 162, 100),
                               (30, 162, 81), (36, 200, 72), (5, 384, 12), (16, 384, 30), (9, 27, 200)])
def test_n2_tiles(g):
    from paper_2110_00733_gb300 import build, hom
    build.build()
    hom.load_library()
    f = ri.random_field(g, 9)
    ref = np.moveaxis(np.fft.rfftn(f, axes=(1, 2, 3)), 0, -1)
    with hom.hom_create(g, np.ones(g), hom.HOM_INPUT_FRACTION_F64, precision=hom.HOM_PREC_FP64) as ctx:
        s = hom.hom_fft_forward(ctx, f)
        assert np.linalg.norm(s - ref) <= 1e-14 * np.linalg.norm(ref)
        back = hom.hom_fft_inverse(ctx, s)
        assert np.linalg.norm(back - f) <= 1e-14 * np.linalg.norm(f)


def test_rate_against_the_runtime_engine():
    """The automatic tile against explicit ones: at 200 faster than 8 columns, which the line engine took and with
    which it was slower than the runtime engine; at 384 the runtime engine's own of four columns."""
    from paper_2110_00733_gb300 import build, hom
    build.build()
    hom.load_library()

    def ms(g, tile2):
        phi = np.random.default_rng(1).random(g).astype(np.float32)
        with hom.hom_create(g, phi, precision=hom.HOM_PREC_FP64, shape=(0, tile2, 0)) as c:
            t = [hom.hom_time_kernels(c, reps=10) for _ in range(5)]
        return min(x["x2_inv"] + x["x2_fwd"] for x in t)

    assert ms((128, 200, 128), 0) <= 0.95 * ms((128, 200, 128), 8)
    assert ms((128, 384, 128), 0) <= 1.02 * ms((128, 384, 128), 4)
