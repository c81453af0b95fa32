"""Deposits of float particles: orders whose warps fall into small boxes, across
mesh faces or anywhere, group remainders and both group sizes, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import mesh
from synth.generators import FOUR_PI_G_ONE
from tests.helpers import rel_rms

pytestmark = pytest.mark.gpu

N = 64
DENSITY_TOL = 1e-5   # float32 deposit vs float64, relative RMS (as tests/test_gpu_mesh.py)


def _positions(n, order, seed=3):
    rng = np.random.default_rng(seed)
    x = (rng.random((n, 3)) * N).astype(np.float32)
    if order == "corner":                      # one cell at the far corner: every upper node wraps
        x = (N - rng.random((n, 3))).astype(np.float32)
    x[x >= N] = 0.0
    if order == "cell":
        c = (x // 4).astype(np.int64)
        x = x[np.argsort(c[:, 0] + 16 * (c[:, 1] + 16 * c[:, 2]), kind="stable")]
    return np.ascontiguousarray(x)


def _pm(mass):
    from paper_1611_01545_gb300 import PM
    return PM(dict(n_fine=N, coarse_ratio=4, tile=16, buffer=8, cmp_ratio=4, vel_bits=16, G=FOUR_PI_G_ONE,
                   mass=mass, count=(0, 0), r_split=6.0 / 4.5, r_cut=6.0))


# 1 .. 65: remainders of a group; 2,490,401: the wide groups (from 152 * 32 * 512 particles)
@pytest.mark.parametrize("order", ["cell", "random", "corner"])
@pytest.mark.parametrize("n", [1, 31, 65, 70001, 2490401])
def test_deposits_of_float_particles(n, order):
    mass = (8.0, 100.0)       # 100 x 2^32 exceeds the int64 bins: corners go to the mesh directly
    pm = _pm(mass)
    x = _positions(n, order)
    xd = torch.from_numpy(x).cuda()
    for s in range(2):
        rc, rf = pm.zeros_meshes()
        pm.deposit(s, xd, rc, rf)
        assert rel_rms(rf.cpu().numpy(), mesh.cic_deposit(x, mass[s], N)) < DENSITY_TOL
        assert rel_rms(rc.cpu().numpy(), mesh.cic_deposit(x / 4.0, mass[s], N // 4)) < DENSITY_TOL
        rc, rf = pm.zeros_meshes(fixed=True)
        pm.deposit_fixed(s, xd, rc, rf)
        M = mesh.fixed_mass(mass[s])
        np.testing.assert_array_equal(rf.cpu().numpy(), mesh.cic_deposit_fixed(x, M, N))
        np.testing.assert_array_equal(rc.cpu().numpy(),
                                      mesh.cic_deposit_fixed((x / np.float32(4)).astype(np.float32), M, N // 4))
    w = np.random.default_rng(4).standard_normal((n, 2)).astype(np.float32)
    w[:, 0] = 1.0
    f = pm.deposit_weights(xd, torch.from_numpy(w).cuda()).cpu().numpy()
    pm.check()
    for q in range(2):
        ref = mesh.cic_deposit(x, w[:, q].astype(np.float64), N)
        scale = np.sqrt(np.mean(mesh.cic_deposit(x, np.abs(w[:, q]).astype(np.float64), N) ** 2))
        assert np.sqrt(np.mean((f[q] - ref) ** 2)) < DENSITY_TOL * scale


# chunks of 2,048 particles: dense (a few cells), sparse (more cells than a chunk keeps), one heavy cell, remainders
@pytest.mark.parametrize("vel_bits", [8, 16])
@pytest.mark.parametrize("n_cdm,heavy", [(1, 0), (700, 0), (2049, 5000), (300007, 9000)])
def test_decompress_chunks(n_cdm, heavy, vel_bits):
    from oracle import codec
    from paper_1611_01545_gb300 import PM
    from tests.helpers import lib_codes_from_oracle
    pm = PM(dict(n_fine=N, coarse_ratio=1, tile=N, buffer=0, cmp_ratio=4, vel_bits=vel_bits, G=FOUR_PI_G_ONE,
                 mass=(8.0, 0.04), count=(0, 0)))
    x = _positions(n_cdm, "random")
    x = np.concatenate([x, np.full((heavy, 3), 33.25, np.float32)])
    v = np.random.default_rng(5).standard_normal(x.shape).astype(np.float32)
    ref = codec.compress(x, v, N, N // 4, vel_bits)
    xd, vd = pm.decompress(0, lib_codes_from_oracle(ref))
    pm.check()
    xr, vr = codec.decompress(ref, N)
    np.testing.assert_array_equal(xd.cpu().numpy(), xr)
    np.testing.assert_array_equal(vd.cpu().numpy(), vr)


# enough particles for the interleaved mesh (half the nodes) against chunks too small for it: the same bits,
# on one stream and on two at once
@pytest.mark.parametrize("n,two", [(32, False), (64, True)])
def test_interleaved_gathers_equal_direct_ones(n, two):
    from paper_1611_01545_gb300 import PM
    cfg = dict(n_fine=n, coarse_ratio=1, tile=n, buffer=0, cmp_ratio=4, vel_bits=16, G=FOUR_PI_G_ONE, mass=(8.0, 0.04),
               count=(0, 0))
    if two:
        cfg.update(coarse_ratio=4, tile=16, buffer=8, r_split=6.0 / 4.5, r_cut=6.0)
    pm = PM(cfg)
    g = torch.Generator(device="cuda").manual_seed(n)
    count = n ** 3 // 2
    x = torch.rand((count, 3), generator=g, device="cuda") * n
    x[:64] = torch.tensor([n - 0.25, 0.0, n - 1.0], device="cuda")       # upper nodes wrap
    v = torch.randn((count, 3), generator=g, device="cuda")
    af = torch.randn((3, n, n, n), generator=g, device="cuda")
    ac = torch.randn((3,) + (n // 4,) * 3, generator=g, device="cuda") if two else None
    chunks = [(i, min(i + 1000, count)) for i in range(0, count, 1000)]
    a = pm.interpolate(x, ac, af)
    assert torch.equal(a, torch.cat([pm.interpolate(x[i:j].contiguous(), ac, af) for i, j in chunks]))
    xk, vk = x.clone(), v.clone()
    pm.kick_drift(xk, vk, ac, af, 0.3, 0.7)
    small = [(x[i:j].clone(), v[i:j].clone()) for i, j in chunks]
    for xs, vs in small:
        pm.kick_drift(xs, vs, ac, af, 0.3, 0.7)
    assert torch.equal(xk, torch.cat([s[0] for s in small])) and torch.equal(vk, torch.cat([s[1] for s in small]))
    streams = [torch.cuda.Stream() for _ in range(2)]
    meshes = [af, -2.0 * af]
    torch.cuda.synchronize()
    got = [[], []]
    for _ in range(5):
        for k, st in enumerate(streams):
            with torch.cuda.stream(st):
                got[k].append(pm.interpolate(x, None if ac is None else (1.0, -2.0)[k] * ac, meshes[k]))
    torch.cuda.synchronize()
    for k, f in enumerate((1.0, -2.0)):
        for r in got[k]:
            assert torch.equal(r, f * a)
    if not two:
        lam = [torch.randn((count, 3), generator=g, device="cuda") for _ in range(2)]
        lx, lv, la = lam[0].clone(), lam[1].clone(), torch.zeros_like(af)
        pm.interpolate_adjoint(x, af, 0.3, 0.7, lx, lv, la)
        parts = [(lam[0][i:j].clone(), lam[1][i:j].clone()) for i, j in chunks]
        for (i, j), (px, pv) in zip(chunks, parts):
            pm.interpolate_adjoint(x[i:j].contiguous(), af, 0.3, 0.7, px, pv, torch.zeros_like(af))
        assert torch.equal(lx, torch.cat([p[0] for p in parts])) and torch.equal(lv, torch.cat([p[1] for p in parts]))
    pm.check()
