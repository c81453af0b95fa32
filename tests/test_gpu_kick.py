"""The recompress passes where they can go wrong: with c_kick = 0 a step is a drift
whose result float32 arithmetic gives exactly, so the new codes must equal the
oracle codec's of the drifted particles bit for bit, in every launch form:
forces staged or gathered directly (dense and sparse sets), rows of 16 to 64
cells and blocks of several rows, every window width, far movers, empty rows,
and cells whose share of a block exceeds the ranks that a key holds."""
import numpy as np
import pytest
import torch

from oracle import codec
from synth.generators import FOUR_PI_G_ONE, fermi_dirac_speeds, isotropic_velocities
from tests.helpers import lib_codes_from_oracle, oracle_codes_from_lib, records

pytestmark = pytest.mark.gpu


def _pm(n, counts, vel_bits, two=True, mode=0):
    from paper_1611_01545_gb300 import PM
    cfg = dict(n_fine=n, coarse_ratio=1, tile=n, buffer=0, cmp_ratio=4, vel_bits=vel_bits, G=FOUR_PI_G_ONE,
               mass=(8.0, 0.04), count=counts, deposit_mode=mode)
    if two:
        cfg.update(coarse_ratio=4, tile=16, buffer=8, r_split=6.0 / 4.5, r_cut=6.0)
    return PM(cfg)


def _species(rng, n, count, speed, vel_bits):
    x = (rng.random((count, 3)) * n).astype(np.float32)
    x[x >= n] = 0.0
    v = isotropic_velocities(rng, fermi_dirac_speeds(rng, count, speed)) if speed else np.zeros((count, 3), np.float32)
    return codec.compress(x, v, n, n // 4, vel_bits)


def _drifted(c, n, vel_bits):
    x, v = codec.decompress(c, n)
    x = (x + v).astype(np.float32)
    x = np.where(x < 0, (x + np.float32(n)).astype(np.float32), x)
    x = np.where(x >= n, (x - np.float32(n)).astype(np.float32), x)
    out = ~((x >= 0) & (x < n))                    # moved more than one box length
    x[out] = x[out] - np.float32(n) * np.floor(x[out] / np.float32(n))
    assert x.dtype == np.float32 and np.all((x >= 0) & (x < n))
    return codec.compress(x, v, n, n // 4, vel_bits)


def _check(pm, codes, n, vel_bits):
    din = [lib_codes_from_oracle(c) for c in codes]
    dout = [pm.empty_codes(c.n, esc_cap=(n // 4) ** 3) for c in codes]
    pm.step(din, dout, 0.0, 1.0)
    pm.check()
    for c, d in zip(codes, dout):
        got, ref = oracle_codes_from_lib(d, n // 4, vel_bits), _drifted(c, n, vel_bits)
        assert got.vmax == ref.vmax
        np.testing.assert_array_equal(got.cnt, ref.cnt)
        np.testing.assert_array_equal(records(got), records(ref))


SHAPES = [None, ((16, 1, 1), 1, 0), ((16, 1, 1), 4, 1), ((8, 1, 1), 2, 0), ((4, 2, 2), 1, 0), ((16, 2, 1), 3, 1),
          ((1, 1, 1), 4, 0)]


# per cell: 0.2 and 9 particles (gathered directly), 20 and 60 (staged); hot and cold
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("counts,speed", [((37, 801), 2.0), ((5000, 32768), 2.0), ((40001, 41999), 0.3),
                                          ((20000, 226000), 6.0), ((0, 90001), 2.0)])
def test_drifted_codes_equal_the_oracle(shape, counts, speed):
    n = 64
    rng = np.random.default_rng(sum(counts))
    for vel_bits, two, mode in ((16, True, 0), (8, True, 1), (8, False, 0)):
        codes = [_species(rng, n, counts[0], 0.05 * speed, vel_bits), _species(rng, n, counts[1], speed, vel_bits)]
        pm = _pm(n, counts, vel_bits, two, mode)
        if shape:
            pm.set_tuning({"kick_block": shape[0], "kick_window": shape[1], "kick_persistent": shape[2]})
        _check(pm, codes, n, vel_bits)


# rows of 48 and of 64 cells, on meshes whose blocks wrap and do not
@pytest.mark.parametrize("n,count", [(192, 1500001), (256, 300001), (256, 3500001)])
def test_long_rows(n, count):
    rng = np.random.default_rng(n)
    codes = [_species(rng, n, count // 9, 0.1, 16), _species(rng, n, count, 2.0, 16)]
    from paper_1611_01545_gb300 import PM
    pm = PM(dict(n_fine=n, coarse_ratio=4, tile=32, buffer=8, cmp_ratio=4, vel_bits=16, G=FOUR_PI_G_ONE,
                 mass=(8.0, 0.04), count=(count // 9, count), r_split=6.0 / 4.5, r_cut=6.0))
    _check(pm, codes, n, 16)


def test_ranks_beyond_the_key():
    # 11 slot bits (16 x 9 x 9 cells) leave 20 rank bits: a cell of 1.2 million particles has more
    n, heavy = 64, 1200000
    rng = np.random.default_rng(8)
    x = np.concatenate([np.full((heavy, 3), 21.5, np.float32) + rng.random((heavy, 3)).astype(np.float32),
                        (rng.random((3000, 3)) * n).astype(np.float32)])
    x[x >= n] = 0.0
    v = (0.2 * rng.standard_normal(x.shape)).astype(np.float32)
    codes = [_species(rng, n, 11, 0.0, 16), codec.compress(x, v, n, n // 4, 16)]
    pm = _pm(n, (11, x.shape[0]), 16)
    pm.set_tuning({"kick_block": (16, 1, 1), "kick_window": 4})
    _check(pm, codes, n, 16)


# a tuning that needs larger tables than the handle holds: with no memory left for
# them the step runs all the same, and a graph captured before keeps its own
@pytest.mark.parametrize("short", [False, True])
def test_tuning_with_larger_tables(short):
    n, counts = 128, (3000, 60000)
    rng = np.random.default_rng(7)
    codes = [_species(rng, n, counts[s], 2.0, 8) for s in range(2)]
    pm = _pm(n, counts, 8)
    din = [lib_codes_from_oracle(c) for c in codes]
    dout = [pm.empty_codes(c.n, esc_cap=(n // 4) ** 3) for c in codes]

    def check():
        torch.cuda.synchronize()
        pm.check()
        for c, d in zip(codes, dout):
            got, ref = oracle_codes_from_lib(d, n // 4, 8), _drifted(c, n, 8)
            assert got.vmax == ref.vmax
            np.testing.assert_array_equal(got.cnt, ref.cnt)
            np.testing.assert_array_equal(records(got), records(ref))
            d.pos.zero_()
            d.cnt.zero_()

    pm.step(din, dout, 0.0, 1.0)
    check()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        pm.step(din, dout, 0.0, 1.0)
    filler = None
    if short:
        torch.cuda.empty_cache()
        free, _ = torch.cuda.mem_get_info()
        filler = torch.empty(free - (100 << 20), dtype=torch.uint8, device="cuda")   # the tables take 191 MB
    tuning = {"kick_block": (1, 1, 1), "kick_window": 4}
    pm.set_tuning(tuning)
    assert pm.get_tuning()["kick_window"] == 4
    pm.step(din, dout, 0.0, 1.0)
    del filler
    torch.cuda.empty_cache()
    check()
    graph.replay()
    check()
