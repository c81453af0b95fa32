"""Coarse and compression ratios other than 4, and launches whose dynamic shared
memory ends just below 48 KB: the fused step against the path of one call per
stage, and drifted codes against the oracle codec."""
import os
import subprocess
import sys

import pytest

from tests import test_gpu_kick as kick
from tests import test_gpu_solve_shapes as shapes

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


# prolongation by 2 and by 8 onto tiles with even buffers, in the library's own launch shapes
@pytest.mark.parametrize("n,ratio,tile,buffer", [(32, 2, 16, 8), (64, 2, 32, 16), (96, 2, 48, 24), (128, 8, 32, 16),
                                                 (128, 8, 64, 16), (384, 8, 96, 16)])
def test_fused_step_ratios(n, ratio, tile, buffer):
    shapes.test_fused_step_solve_shapes(n, ratio, tile, buffer)


def _deposit_edge():
    # blocks of 16 x 1 x 1 cells of 8 fine cells: 49,072 bytes of bins and offsets
    shapes.test_fused_step_solve_shapes(128, 8, 32, 16)


def _kick_edge(n, block, window):
    counts = (3000, 60000)
    rng = kick.np.random.default_rng(n)
    codes = [kick._species(rng, n, c, 2.0, 16) for c in counts]
    pm = kick._pm(n, counts, 16)
    pm.set_tuning({"kick_block": block, "kick_window": window})
    kick._check(pm, codes, n, 16)


def _count_edge():
    _kick_edge(128, (16, 2, 1), 3)       # 49,064 bytes


def _scatter_edge():
    _kick_edge(192, (48, 2, 2), 3)       # 49,152 bytes


# Dynamic shared memory of at most 48 KB that exceeds them together with the
# kernel's static part.  Each in a process of its own: a larger launch of the same
# kernel earlier in the process would have raised its limit.
@pytest.mark.parametrize("edge", ["_deposit_edge", "_count_edge", "_scatter_edge"])
def test_shared_memory_edge(edge):
    code = f"from tests import test_gpu_ratios as t; t.{edge}()"
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
