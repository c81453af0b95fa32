"""The tile and mesh solves over every transform size and window shape against the
oracle: odd buffers (window rows that do not pair with output rows), tiles of two
cells, 96^3 windows on and off 16-cell boundaries, few and many output row pairs,
integer densities, single meshes, and the fused step with the coarse force
prolonged onto the tiles by 2 and by 4."""
import numpy as np
import pytest
import torch

from oracle import codec, solve
from tests.helpers import assert_codes_match, lib_codes_from_oracle, oracle_codes_from_lib, rel_rms

pytestmark = pytest.mark.gpu

MESH_ACC_TOL = 1e-5   # as tests/test_gpu_mesh.py
G = 1 / (4 * np.pi)

# n, coarse ratio, tile, buffer
TILES = [(32, 2, 2, 7), (32, 2, 16, 8), (64, 4, 16, 8), (64, 2, 32, 16), (96, 2, 6, 21), (96, 2, 48, 8),
         (96, 2, 24, 36), (192, 4, 64, 16), (192, 4, 48, 24), (192, 4, 96, 16)]


def _cfg(n, ratio, tile, buffer, **kw):
    cut = float(buffer - 2)
    return dict(n_fine=n, coarse_ratio=ratio, tile=tile, buffer=buffer, cmp_ratio=ratio, vel_bits=16, G=G,
                mass=(8.0, 0.5), count=(0, 0), r_split=cut / 4.5, r_cut=cut, **kw)


def _density(n, fixed, seed):
    rng = np.random.default_rng(seed)
    rho = rng.random((n, n, n)) * 4.0
    if fixed:
        q = np.round(rho * 2.0 ** 32).astype(np.int64)
        return torch.from_numpy(q), q.astype(np.float64) / 2.0 ** 32
    f = rho.astype(np.float32)
    return torch.from_numpy(f), f.astype(np.float64)


def _tile_accel(rho, cfg, idx):
    t, b = cfg["tile"], cfg["buffer"]
    i = np.arange(t + 2 * b)
    w = [(k * t - b + i) % cfg["n_fine"] for k in idx]
    K = solve.fine_kernel(t + 2 * b, cfg["G"], cfg["r_split"], cfg["r_cut"])
    return solve.accel_tile(rho[np.ix_(w[2], w[1], w[0])], K)[:, b:b + t, b:b + t, b:b + t]


@pytest.mark.parametrize("n,ratio,tile,buffer", TILES)
@pytest.mark.parametrize("fixed", [False, True])
def test_tile_solve_shapes(n, ratio, tile, buffer, fixed):
    from paper_1611_01545_gb300 import PM
    cfg = _cfg(n, ratio, tile, buffer, deposit_mode=int(fixed))
    pm = PM(cfg)
    rf, ref_f = _density(n, fixed, n + tile)
    rc, ref_c = _density(n // ratio, fixed, n + tile + 1)
    ac, af = pm.zeros_acc()
    pm.solve(rc.cuda(), rf.cuda(), ac, af)
    pm.check()
    assert rel_rms(ac.cpu().numpy(), solve.accel_periodic(ref_c, float(ratio), G, cfg["r_split"])) < MESH_ACC_TOL
    last, af = n // tile - 1, af.cpu().numpy()
    for idx in {(0, 0, 0), (last, 0, last // 2), (last, last, last)}:
        x, y, z = (k * tile for k in idx)
        got = af[:, z:z + tile, y:y + tile, x:x + tile]
        assert rel_rms(got, _tile_accel(ref_f, cfg, idx)) < MESH_ACC_TOL, idx


@pytest.mark.parametrize("n", [16, 32, 48, 64, 96, 128])
@pytest.mark.parametrize("fixed", [False, True])
def test_single_mesh_solve_shapes(n, fixed):
    from paper_1611_01545_gb300 import PM
    pm = PM(dict(n_fine=n, coarse_ratio=1, tile=n, buffer=0, cmp_ratio=4, vel_bits=16, G=G, mass=(1.0, 1.0),
                 deposit_mode=int(fixed)))
    rf, ref = _density(n, fixed, n)
    _, af = pm.zeros_acc()
    pm.solve(None, rf.cuda(), None, af)
    pm.check()
    assert rel_rms(af.cpu().numpy(), solve.accel_periodic(ref, 1.0, G)) < MESH_ACC_TOL


# prolongation by 2 (odd buffers) and 4, against the path of one call per stage
@pytest.mark.parametrize("n,ratio,tile,buffer", [(32, 2, 2, 7), (64, 4, 16, 8), (64, 4, 4, 14),
                                                 (96, 2, 6, 21), (192, 4, 64, 16)])
def test_fused_step_solve_shapes(n, ratio, tile, buffer):
    from paper_1611_01545_gb300 import PM
    rng = np.random.default_rng(n + ratio + tile)
    codes = []
    for count in (500, 4000):
        x = (rng.random((count, 3)) * n).astype(np.float32)
        x[x >= n] = 0.0
        codes.append(codec.compress(x, (rng.standard_normal((count, 3)) * 0.3).astype(np.float32), n, n // ratio, 8))
    pm = PM(dict(_cfg(n, ratio, tile, buffer), vel_bits=8, count=tuple(c.n for c in codes)))
    dout = [pm.empty_codes(c.n, esc_cap=64) for c in codes]
    pm.step([lib_codes_from_oracle(c) for c in codes], dout, 0.5, 1.0)
    pm.check()
    rc, rf = pm.zeros_meshes()
    xv = [[torch.from_numpy(a).cuda() for a in codec.decompress(c, n)] for c in codes]
    for s in range(2):
        pm.deposit(s, xv[s][0], rc, rf)
    ac, af = pm.zeros_acc()
    pm.solve(rc, rf, ac, af)
    for s in range(2):
        pm.kick_drift(*xv[s], ac, af, 0.5, 1.0)
        plain = pm.compress(s, *xv[s])
        pm.check()
        got, ref = (oracle_codes_from_lib(c, n // ratio, 8) for c in (dout[s], plain))
        assert abs(float(got.vmax) - float(ref.vmax)) <= 1e-5 * float(ref.vmax)
        assert_codes_match(got, ref, f"{n} / {tile} + {buffer} species {s}")
