"""The debug build (kernel indices checked, a status for any outside its buffer) on the kernels that only odd-Nx boxes
without padding reach: the one-node kernels of the FP32-arithmetic forms and a batch's one-node single pass."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import test_gpu_tiled as t
for prec in ("f32", "f16"):
    for op in ("nonorth", "orth", "nonorth_d3q15"):
        t._assert_tiled(t._fields(t.ODD, op, prec, t._tile(t.ODD), t.ODD_COPIES, 2),
                        t._fields(t.ODD, op, prec, t._tile(t.ODD), (1, 1, 1), 2))
    for grid in ((5, 6144, 6300), (511, 33000, 3)):
        t._batch(prec, grid, [(16, 12, 10), (15, 12, 10)])
print("no index outside")
"""


def test_debug_build_on_unpadded_rows():
    from paper_1805_08643_gb300 import _build

    _build.build(debug=True)
    r = subprocess.run([sys.executable, "-c", CODE.format(root=ROOT, tests=os.path.join(ROOT, "tests"))],
                       capture_output=True, text=True, timeout=600, cwd=ROOT,
                       env=dict(os.environ, LBM_DEBUG_LIBRARY="1"))
    assert r.returncode == 0 and "no index outside" in r.stdout, r.stderr[-3000:]
