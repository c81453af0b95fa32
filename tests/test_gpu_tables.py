"""Memory of the recompress passes' start tables: a mesh with few particles does not
take tables larger than its bound, and a handle with no room for them still
steps, with the codes that the oracle gives."""
import numpy as np
import pytest
import torch

from oracle import codec
from synth.generators import FOUR_PI_G_ONE
from tests.helpers import lib_codes_from_oracle, oracle_codes_from_lib, records

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _cfg(n, ratio, tile, buffer, counts):
    cut = float(buffer - 2)
    return dict(n_fine=n, coarse_ratio=ratio, tile=tile, buffer=buffer, cmp_ratio=ratio, vel_bits=8, G=FOUR_PI_G_ONE,
                mass=(8.0, 0.04), count=counts, r_split=cut / 4.5, r_cut=cut, tile_batch=64)


def _codes(n, ratio, counts, seed):
    rng = np.random.default_rng(seed)
    out = []
    for c in counts:
        x = (rng.random((c, 3)) * n).astype(np.float32)
        x[x >= n] = 0.0
        out.append(codec.compress(x, (2.0 * rng.standard_normal((c, 3))).astype(np.float32), n, n // ratio, 8))
    return out


def _drift_matches(pm, codes, n, ratio):
    """A step with c_kick = 0 gives the oracle codec's codes of the drifted particles."""
    din = [lib_codes_from_oracle(c) for c in codes]
    dout = [pm.empty_codes(c.n, esc_cap=64) for c in codes]
    pm.step(din, dout, 0.0, 1.0)
    pm.check()
    for c, d in zip(codes, dout):
        x, v = codec.decompress(c, n)
        x = (x + v).astype(np.float32)
        x = np.where(x < 0, (x + np.float32(n)).astype(np.float32), x)
        x = np.where(x >= n, (x - np.float32(n)).astype(np.float32), x)
        assert np.all((x >= 0) & (x < n))
        ref, got = codec.compress(x, v, n, n // ratio, 8), oracle_codes_from_lib(d, n // ratio, 8)
        assert got.vmax == ref.vmax
        np.testing.assert_array_equal(got.cnt, ref.cnt)
        np.testing.assert_array_equal(records(got), records(ref))


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_tables_of_a_sparse_mesh_are_bounded():
    """192^3 compression cells: windows of half-width 1 take 531 MB of tables, more
    than the bound of a handle for a thousand particles (256 MB), less than that
    of one for 40 million (their scratch of 20 bytes each)."""
    from paper_1611_01545_gb300 import PM
    took = []
    for counts in ((500, 500), (500, 40000000)):
        before = _free()
        pm = PM(_cfg(768, 4, 64, 16, counts))
        took.append(before - _free() - 20 * sum(counts))
        if counts[1] == 500:
            _drift_matches(pm, _codes(768, 4, counts, 2), 768, 4)
        pm.close()
    assert took[1] - took[0] > 400 * MB


def test_mesh_with_no_tables_at_all():
    """384^3 compression cells and a thousand particles: even the blocks' own cells
    exceed the bound, so every particle is counted on its own."""
    from paper_1611_01545_gb300 import PM
    counts = (500, 500)
    pm = PM(_cfg(768, 2, 64, 16, counts))
    _drift_matches(pm, _codes(768, 2, counts, 3), 768, 2)


# 128^3 compression cells: 144 MB of tables (rows of 128 cells, 9 rows of windows, 8
# bytes), 16 MB with windows of the blocks' own cells: room for the latter, and for neither
@pytest.mark.parametrize("short_mb", [60, 136])
def test_handle_with_no_room_for_tables(short_mb):
    from paper_1611_01545_gb300 import PM
    n, ratio, counts = 256, 2, (3000, 60000)
    codes = _codes(n, ratio, counts, 4)
    cfg = _cfg(n, ratio, 64, 16, counts)
    pm = PM(cfg)
    _drift_matches(pm, codes, n, ratio)       # kernels loaded
    pm.close()
    before = _free()
    pm = PM(cfg)
    need = before - _free()
    pm.close()
    filler = torch.empty(_free() - need + short_mb * MB, dtype=torch.uint8, device="cuda")
    try:
        pm = PM(cfg)
    finally:
        del filler
        torch.cuda.empty_cache()
    _drift_matches(pm, codes, n, ratio)
