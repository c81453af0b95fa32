"""Memory of the recompress passes' start tables: the autotuner gives back what
its candidates took and never picks a shape whose tables cannot be had, a mesh
with few particles does not take tables larger than its bound, and a handle
with no room for them still steps, with the codes that the oracle gives."""
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


def _table(n_cmp, tuning):
    """Bytes of the tables of a tuning: a word per block, species and window cell."""
    window = blocks = 1
    for r in tuning["kick_block"]:
        window *= min(r + 2 * tuning["kick_window"], n_cmp)
        blocks *= n_cmp // r
    return 8 * window * blocks


def test_autotune_gives_its_tables_back():
    from paper_1611_01545_gb300 import PM
    n, counts = 256, (3000, 60000)
    codes = _codes(n, 4, counts, 1)
    cfg = _cfg(n, 4, 64, 16, counts)
    pm = PM(cfg)
    din = [lib_codes_from_oracle(c) for c in codes]
    dout = [pm.empty_codes(c.n, esc_cap=64) for c in codes]
    pm.step(din, dout, 0.0, 1.0)
    before = _free()
    chosen = pm.autotune(din, dout, 0.0, 1.0, reps=1)
    # beside the chosen shape's tables only what the kernels used for the first time take to load
    assert before - _free() <= _table(n // 4, chosen) + 48 * MB
    _drift_matches(pm, codes, n, 4)
    pm.close()
    # with 40 MB left, shapes whose tables exceed that and what pm_init reserved are no candidates
    pm = PM(cfg)
    held = _table(n // 4, pm.get_tuning())
    pm.step(din, dout, 0.0, 1.0)
    filler = torch.empty(_free() - 40 * MB, dtype=torch.uint8, device="cuda")
    for _ in range(5):
        chosen = pm.autotune(din, dout, 0.0, 1.0, reps=1)
        assert _table(n // 4, chosen) <= held + 40 * MB
    del filler
    torch.cuda.empty_cache()
    _drift_matches(pm, codes, n, 4)


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
