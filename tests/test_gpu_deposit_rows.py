"""The fused float deposit of cell-row blocks against the oracle: every row length,
one and two rows per block, blocks that wrap and meshes of one block, empty and
heavy cells, empty species, sparse and dense sets, a density mesh that is not
16-byte aligned (the general kernel), and a non-zero mesh to add to."""
import numpy as np
import pytest
import torch

from oracle import codec, mesh
from synth.generators import FOUR_PI_G_ONE
from tests.helpers import lib_codes_from_oracle, rel_rms

pytestmark = pytest.mark.gpu

DENSITY_TOL = 1e-5   # as tests/test_gpu_mesh.py
MASS = (8.0, 0.04)


def _set(n, count, heavy, seed):
    rng = np.random.default_rng(seed)
    x = (rng.random((count, 3)) * n).astype(np.float32)
    if heavy:
        x = np.concatenate([x, (np.array([n - 4, 4, n - 4]) + 4 * rng.random((heavy, 3))).astype(np.float32)])
    x[x >= n] = 0.0
    return codec.compress(x, np.zeros_like(x), n, n // 4, 8)


# rows of 1 to 64 cells, one and two of them per block
@pytest.mark.parametrize("n,shape", [(64, (16, 1, 1)), (64, (8, 2, 1)), (64, (1, 1, 1)), (64, (2, 2, 1)),
                                     (128, (32, 1, 1)), (128, (32, 2, 1)), (192, (48, 1, 1)), (192, (24, 2, 1)),
                                     (256, (64, 1, 1)), (256, (32, 2, 1))])
@pytest.mark.parametrize("counts", [(0, 300), (9000, 70000), (3, 0)])
def test_deposit_rows(n, shape, counts):
    from paper_1611_01545_gb300 import PM
    pm = PM(dict(n_fine=n, coarse_ratio=4, tile=16 if n == 64 else 32, buffer=8, cmp_ratio=4, vel_bits=8,
                 G=FOUR_PI_G_ONE, mass=MASS, count=(0, 0), r_split=6.0 / 4.5, r_cut=6.0))
    codes = [_set(n, counts[s], 700 * s if counts[s] > 3 else 0, 10 * n + s) for s in range(2)]
    xs = [codec.decompress(c, n)[0] for c in codes]
    ref_f = 1.5 + sum(mesh.cic_deposit(x, MASS[s], n) for s, x in enumerate(xs))
    ref_c = 2.5 + sum(mesh.cic_deposit(x / 4.0, MASS[s], n // 4) for s, x in enumerate(xs))
    dc = [lib_codes_from_oracle(c) for c in codes]
    for persistent in (0, 1):
        pm.set_tuning({"deposit_block": shape, "deposit_persistent": persistent})
        for shift in (0, 1):
            rf = torch.full((n ** 3 + 4,), 1.5, device="cuda")[shift:shift + n ** 3].view(n, n, n)
            rc = torch.full((n // 4,) * 3, 2.5, device="cuda")
            pm.deposit_codes(dc, rc, rf)
            pm.check()
            assert rel_rms(rf.cpu().numpy(), ref_f) < DENSITY_TOL
            assert rel_rms(rc.cpu().numpy(), ref_c) < DENSITY_TOL
