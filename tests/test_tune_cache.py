"""The autotuner's file: shapes timed on these kernels are taken from it, without any device work;
lines of other kernels (and the lines without a name, which earlier versions wrote) are not."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import ctypes
from paper_2110_00733_gb300 import hom
shape = (ctypes.c_int * 3)(-1, -1, -1)
rc = hom.load_library().hom_autotune((ctypes.c_int * 3)(18, 16, 20), 0, shape)
print(rc, *shape)
"""


@pytest.mark.parametrize("lines, taken", [
    (["k2 18 16 20 0 3 4 5"], True),
    (["16 16 16 0 1 8 1", "k1 18 16 20 0 9 9 9", "k2 18 16 20 0 3 4 5"], True),
    (["18 16 20 0 3 4 5"], False),
    (["k1 18 16 20 0 3 4 5", "k2 18 16 24 0 3 4 5", "k2 18 16 20 1 3 4 5", "k2 18 16 20 0 3 4"], False),
])
def test_lines_of_these_kernels_only(tmp_path, lines, taken):
    from paper_2110_00733_gb300 import build
    build.build()
    cache = tmp_path / "tuned"
    cache.write_text("\n".join(lines) + "\n")
    # no device is visible, so that a grid that is not in the file ends in an error and not in a measurement
    env = dict(os.environ, HOM_TUNE_CACHE=str(cache), CUDA_VISIBLE_DEVICES="", PYTHONPATH=ROOT)
    out = subprocess.run([sys.executable, "-c", CODE], env=env, capture_output=True, text=True, check=True, cwd=ROOT).stdout
    rc, *shape = map(int, out.split())
    assert (rc == 0 and shape == [3, 4, 5]) if taken else (rc < 0 and shape == [-1, -1, -1])
