"""Cell-count scans at their edges: cell counts that are no multiple of a thread's
8 cells, one and many tiles, count bytes at any alignment, escapes in every
tile, and launch after launch on one handle, against the oracle codec."""
import numpy as np
import pytest
import torch

from oracle import codec
from tests.helpers import lib_codes_from_oracle, oracle_codes_from_lib, records

pytestmark = pytest.mark.gpu


def _pm(n_fine, cmp_ratio):
    from paper_1611_01545_gb300 import PM
    return PM(dict(n_fine=n_fine, coarse_ratio=1, tile=n_fine, buffer=0, cmp_ratio=cmp_ratio, vel_bits=16,
                   G=1 / (4 * np.pi), mass=(8.0, 0.04), count=(0, 0)))


def _set(n_fine, cmp_ratio, n, heavy, seed):
    rng = np.random.default_rng(seed)
    x = (rng.random((n, 3)) * n_fine).astype(np.float32)
    x[x >= n_fine] = 0.0
    at = (rng.random((heavy, 3)) * n_fine).astype(np.float32)        # cells of 300 particles and more
    at[at >= n_fine] = 0.0
    x = np.concatenate([x, np.repeat(at, 300, axis=0)])
    return x, rng.standard_normal(x.shape).astype(np.float32)


# (n_fine, cmp_ratio): 27, 512, 4096, 32768 (16 tiles) and 110592 (54 tiles) cells
@pytest.mark.parametrize("n_fine,cmp_ratio", [(48, 16), (16, 2), (64, 4), (128, 4), (96, 2)])
@pytest.mark.parametrize("shift", [0, 3])
def test_scans_match_the_codec(n_fine, cmp_ratio, shift):
    pm, nc = _pm(n_fine, cmp_ratio), n_fine // cmp_ratio
    for seed in range(3):
        x, v = _set(n_fine, cmp_ratio, 5000 * seed, 40, seed)
        ref = codec.compress(x, v, n_fine, nc, 16)
        assert ref.esc_cell.size > 0
        dc = lib_codes_from_oracle(ref)
        moved = torch.empty(nc ** 3 + 8, dtype=torch.uint8, device="cuda")
        moved[shift:shift + nc ** 3] = dc.cnt
        dc.cnt = moved[shift:shift + nc ** 3]
        xd, vd = pm.decompress(0, dc)
        pm.check()
        xr, vr = codec.decompress(ref, n_fine)
        np.testing.assert_array_equal(xd.cpu().numpy(), xr)
        np.testing.assert_array_equal(vd.cpu().numpy(), vr)
        out = pm.empty_codes(x.shape[0], esc_cap=ref.esc_cell.size)
        out.cnt = torch.empty(nc ** 3 + 8, dtype=torch.uint8, device="cuda")[shift:shift + nc ** 3]
        got = pm.compress(0, torch.from_numpy(x).cuda(), torch.from_numpy(v).cuda(), out=out)
        pm.check()
        g = oracle_codes_from_lib(got, nc, 16)
        np.testing.assert_array_equal(g.cnt, ref.cnt)
        np.testing.assert_array_equal(g.esc_cell, ref.esc_cell)
        np.testing.assert_array_equal(g.esc_count, ref.esc_count)
        np.testing.assert_array_equal(records(g), records(ref))
