"""What a program that steps a two-species particle-mesh simulation has this
framework do, as cases that can be timed and compared.

Kinds of case (the "kind" of a case dict):

  step     two fused steps a -> b -> c over the compressed state (pm.step, each
           reading the other's codes) and the density of the state reached
           (pm.deposit_codes).  The order of the records inside a compression
           cell is unspecified, so the state reached is handed back as what it
           is used for next: both density meshes and the species' v_max.  The
           second step makes them depend on the first one's velocity codes.
  solve    density meshes in, acceleration meshes out (pm.solve).
  deposit  codes in, density meshes out (pm.deposit_codes): a step's first half.
  plain    one step over float particles (pm.step_plain), as the uncompressed
           arm of the compression study and every differentiable forward run it.
  reverse  one step of a differentiable trajectory and its reverse step
           (pm.step_plain, pm.step_adjoint with the kept force mesh).
  restart  a float state compressed and decompressed, and the number and
           momentum density of what comes back (the study's restart arm).
  pp       Eq. 4 accelerations of every particle (pm.pp_accel).

Meshes, tiles, species counts (8 neutrinos per CDM particle), masses, the
Zel'dovich / lognormal / Fermi-Dirac recipes and the launch tuning of the large
cases are those of this repository's workloads (synth/, bench.py); particle
counts with odd sides stand beside its powers of two.
"""
import math

import numpy as np
import torch

from paper_1611_01545_gb300 import PM
from paper_1611_01545_gb300.pm import Codes

MASS = (8.0, 0.04)              # CDM, neutrino (ratio 0.005)
G = 1.0 / (4.0 * math.pi)       # 4 pi G = 1
FD_SCALE = 2.0                  # neutrino speeds |v| = 2 u, u Fermi-Dirac
R = 4                           # fine cells per coarse and per compression cell
KICK = 2.0 ** -14               # c_kick of the compressed steps: an early step, in which thermal motion moves the
                                # neutrinos by cells while gravity changes velocities little

# (n_fine, tile, buffer); tile 0: one periodic mesh.  Tile edges T = tile + 2 buffer of 32 to 128.
SMALL = [(32, 0, 0), (48, 0, 0), (64, 0, 0), (96, 0, 0), (128, 0, 0),
         (64, 16, 8), (128, 32, 16), (128, 64, 16), (192, 32, 8)]
MEDIUM = [(192, 64, 16), (192, 96, 16), (256, 32, 16), (256, 64, 16), (384, 64, 16), (384, 96, 16)]
LARGE = [(512, 64, 16), (768, 64, 16), (768, 96, 16)]

# The shapes a tuned program keeps on the large meshes (bench.py's tuning of the largest workload).
TUNING = {"deposit_block": [32, 2, 1], "deposit_persistent": 1, "kick_block": [64, 1, 1], "kick_window": 1,
          "kick_persistent": 0}


def _case(kind, geometry, n_cdm, n_nu, **more):
    n, tile, buffer = geometry
    c = {"kind": kind, "n_fine": n, "tile": tile, "buffer": buffer, "n_cdm": n_cdm, "n_nu": n_nu, "vel_bits": 16,
         "cdm": "zeldovich", "c_kick": KICK, "c_drift": 1.0, "tuned": False, "graphs": False}
    c.update(more)
    return c


def listed():
    return [
        # the smallest run: one periodic 64^3 mesh, 36,864 particles; latency and launches
        dict(_case("step", (64, 0, 0), 16, 32), name="step_mesh64"),
        # a small two-level run with odd particle counts and 48^3 tiles
        dict(_case("step", (192, 32, 8), 33, 65, c_drift=0.25), name="step_tiles192_odd"),
        # the 256^3 workload: 8-bit velocities, tuned, replayed from a graph
        dict(_case("step", (256, 64, 16), 128, 256, vel_bits=8, tuned=True, graphs=True), name="step_tiles256_u8"),
        # the clustered 512^3 workload: lognormal CDM, very uneven cells, the library's own launch shapes
        dict(_case("step", (512, 64, 16), 256, 512, cdm="lognormal", c_drift=0.25), name="step_clustered512"),
        # production: an eighth of the largest one-GPU workload at its own density and tuning
        dict(_case("step", (768, 64, 16), 384, 768, tuned=True), name="step_tiles768"),
        # the force solve by itself: 64 tiles of 96^3 and the 64^3 coarse mesh
        dict(_case("solve", (256, 64, 16), 0, 0), name="solve_tiles256"),
        # the largest single periodic mesh
        dict(_case("solve", (128, 0, 0), 0, 0), name="solve_mesh128"),
        # the density of a compressed state alone (diagnostics, a step's first half)
        dict(_case("deposit", (256, 64, 16), 128, 256), name="deposit_tiles256"),
        # an uncompressed step, particles in the cell order that decompression leaves
        dict(_case("plain", (256, 64, 16), 128, 256, c_kick=0.25, c_drift=0.25, order="cell"), name="plain_tiles256"),
        # one step of the differentiable 128^3 run and its reverse step
        dict(_case("reverse", (128, 0, 0), 64, 128, c_kick=0.25, c_drift=0.25, order="random"), name="reverse_mesh128"),
        # the compression study's restart of a 256^3 state in its initial (lattice / random) order
        dict(_case("restart", (256, 64, 16), 128, 256, order="random"), name="restart_tiles256"),
        # the particle-particle option on the 256^3 workload
        dict(_case("pp", (256, 64, 16), 128, 256, vel_bits=8), name="pp_tiles256"),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "solve", "deposit", "plain", "reverse", "restart", "pp"])
    if kind == "step":
        geometry = rng.choice(rng.choice([SMALL, MEDIUM, LARGE]))
    elif kind in ("solve", "deposit"):
        geometry = rng.choice(rng.choice([SMALL, MEDIUM]))
    elif kind == "reverse":
        geometry = rng.choice(SMALL[:5])
    elif kind == "pp":
        geometry = rng.choice(SMALL[5:] + MEDIUM[:4])
    else:
        geometry = rng.choice(SMALL + MEDIUM[:4])
    n = geometry[0]
    n_nu = int(round(n * math.exp(rng.uniform(math.log(0.4), 0.0))))
    n_cdm = max(4, n_nu // 2)
    if kind in ("plain", "reverse", "restart"):
        n_nu = min(n_nu, 256)
    c = _case(kind, geometry, n_cdm, n_nu, vel_bits=rng.choice([8, 16]), cdm=rng.choice(["zeldovich", "lognormal"]),
              c_drift=rng.choice([0.25, 1.0]))
    if kind == "step":
        c["tuned"] = geometry[1] > 0 and (n // R) % 64 == 0 and rng.random() < 0.5
        c["graphs"] = rng.random() < 0.3
    if kind in ("plain", "reverse"):
        c["c_kick"] = c["c_drift"] = 0.25
    if kind in ("plain", "reverse", "restart"):
        c["order"] = rng.choice(["cell", "random"])
    if kind == "pp":
        c["cdm"] = "zeldovich"
    return c


def _r_cut(case):
    return float(case["buffer"] - 2)


def _config(case):
    n = case["n_fine"]
    cfg = {"n_fine": n, "coarse_ratio": 1, "cmp_ratio": R, "vel_bits": case["vel_bits"], "G": G, "mass": MASS,
           "count": (case["n_cdm"] ** 3, case["n_nu"] ** 3)}
    if case["tile"]:
        cfg.update(coarse_ratio=R, tile=case["tile"], buffer=case["buffer"], r_cut=_r_cut(case),
                   r_split=_r_cut(case) / 4.5)
        if case["tuned"]:
            cfg["tile_batch"] = 256
    if case["kind"] == "pp":
        cfg.update(pp=1, r_soft=n / (20.0 * case["n_cdm"]))
    return cfg


# ---- inputs, from the seed alone ------------------------------------------

def _field(g, n, slope, smooth=0.0):
    """Fourier modes of a Gaussian random field on n^3 with P(k) ~ k^slope, and its wave numbers."""
    dk = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device="cuda"))
    k = torch.fft.fftfreq(n, device="cuda") * 2 * math.pi
    kx = torch.fft.rfftfreq(n, device="cuda") * 2 * math.pi
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kx[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    dk *= k2 ** (slope / 4.0) * torch.exp(-0.5 * k2 * smooth * smooth)
    dk[0, 0, 0] = 0.0
    return dk, k2, (kx[None, None, :], k[None, :, None], k[:, None, None])


def _wrap(x, n):
    x = torch.remainder(x, float(n))
    return torch.where(x >= n, torch.zeros_like(x), x)


def _cdm(g, case):
    """CDM positions and velocities: lattice + Zel'dovich displacement, or a lognormal density."""
    n, side = case["n_fine"], case["n_cdm"]
    if case["cdm"] == "lognormal":
        grid = max(8, n // 4)
        f = torch.fft.irfftn(_field(g, grid, -2.0, 1.0)[0], s=(grid,) * 3)
        f = f / f.std()
        cdf = torch.cumsum(torch.exp(1.5 * f.double()).reshape(-1), 0)
        u = torch.rand(side ** 3, generator=g, device="cuda", dtype=torch.float64) * cdf[-1]
        cell = torch.searchsorted(cdf, u).clamp_(max=grid ** 3 - 1)
        q = torch.stack([cell % grid, (cell // grid) % grid, cell // (grid * grid)], dim=1).float()
        x = (q + torch.rand((side ** 3, 3), generator=g, device="cuda")) * (n / grid)
        return _wrap(x, n), 0.05 * torch.randn((side ** 3, 3), generator=g, device="cuda")
    dk, k2, ks = _field(g, side, -2.0)
    psi = torch.stack([torch.fft.irfftn(1j * k * dk / k2, s=(side,) * 3).reshape(-1) for k in ks], dim=1)
    psi *= 0.5 / psi.square().sum(1).mean().sqrt()
    q = (torch.arange(side, device="cuda") + 0.5) * (n / side)
    x = psi.clone()
    x[:, 0] += q.repeat(side * side)
    x[:, 1] += q.repeat_interleave(side).repeat(side)
    x[:, 2] += q.repeat_interleave(side * side)
    return _wrap(x, n), psi * 0.1


def _fermi_dirac():
    """Quantiles of p(u) ~ u^2 / (e^u + 1) on a uniform grid of 65,536 probabilities."""
    u = np.linspace(0.0, 40.0, 8193)
    pdf = u * u / (np.exp(u) + 1.0)
    cdf = np.concatenate([[0.0], np.cumsum(0.5 * (pdf[1:] + pdf[:-1]))])
    p = (np.arange(65536) + 0.5) / 65536
    return torch.from_numpy((FD_SCALE * np.interp(p, cdf / cdf[-1], u)).astype(np.float32)).cuda()


def _hot(g, n, table):
    """Isotropic velocities with Fermi-Dirac speeds."""
    d = torch.randn((n, 3), generator=g, device="cuda")
    speed = table[torch.randint(65536, (n,), generator=g, device="cuda")]
    return d.mul_((speed / d.square().sum(1).sqrt_().clamp_min_(1e-20))[:, None])


def _vel_codes(v, vmax, bits, out):
    half = 1 << (bits - 1)
    q = torch.floor(v * (half / vmax) + half).clamp_(0, 2 * half - 1).int()
    out[:, :3] = torch.where(q > 32767, q - 65536, q).to(torch.int16) if bits == 16 else q.to(torch.uint8)


def _codes_of_counts(count, n, n_cmp, bits):
    c = Codes.empty(n, n_cmp, bits)
    c.cnt.copy_(count.clamp(max=255).to(torch.uint8))
    big = torch.nonzero(count >= 255).reshape(-1)
    if big.numel():
        c.esc[:big.numel(), 0] = big.int()
        c.esc[:big.numel(), 1] = count[big].int()
    c.n_esc.fill_(big.numel())
    return c


def _encode(x, v, n_cmp, bits):
    """Codes of float particles, in cell order."""
    u = x / R
    c = u.floor().clamp_(max=n_cmp - 1)
    q = ((u - c) * 256).clamp_(max=255).to(torch.uint8)
    c = c.int()
    cell, order = torch.sort(c[:, 0] + n_cmp * (c[:, 1] + n_cmp * c[:, 2]), stable=True)
    codes = _codes_of_counts(torch.bincount(cell, minlength=n_cmp ** 3), x.shape[0], n_cmp, bits)
    codes.pos[:, :3] = q[order]
    codes.vmax.copy_(v.abs().max())
    _vel_codes(v[order], codes.vmax, bits, codes.vel)
    return codes


def _neutrino_codes(g, n, n_cmp, bits):
    """Codes of uniform hot neutrinos, drawn cell by cell: uniform offsets, Fermi-Dirac velocities."""
    count = torch.zeros(n_cmp ** 3, dtype=torch.int64, device="cuda")
    chunk, table = 1 << 26, _fermi_dirac()
    parts = [(i, min(i + chunk, n)) for i in range(0, n, chunk)]
    for i, j in parts:
        count += torch.bincount(torch.randint(n_cmp ** 3, (j - i,), generator=g, device="cuda"), minlength=n_cmp ** 3)
    codes = _codes_of_counts(count, n, n_cmp, bits)
    codes.vmax.fill_(40.0)
    for i, j in parts:
        codes.pos[i:j, :3] = torch.randint(256, (j - i, 3), generator=g, device="cuda", dtype=torch.uint8)
        _vel_codes(_hot(g, j - i, table), codes.vmax, bits, codes.vel[i:j])
    return codes


def _codes(g, case):
    n_cmp = case["n_fine"] // R
    x, v = _cdm(g, case)
    return [_encode(x, v, n_cmp, case["vel_bits"]), _neutrino_codes(g, case["n_nu"] ** 3, n_cmp, case["vel_bits"])]


def _particles(g, case):
    n, count = case["n_fine"], case["n_nu"] ** 3
    x, v = _cdm(g, case)
    xn = _wrap(torch.rand((count, 3), generator=g, device="cuda") * n, n)
    xs, vs = [x, xn], [v, _hot(g, count, _fermi_dirac())]
    if case["order"] == "cell":
        for s in range(2):
            c = (xs[s] / R).int()
            order = torch.argsort(c[:, 0] + (n // R) * (c[:, 1] + (n // R) * c[:, 2]), stable=True)
            xs[s], vs[s] = xs[s][order].contiguous(), vs[s][order].contiguous()
    return xs, vs


def _densities(g, case):
    """A clustered density on the fine mesh and what of it the coarse mesh holds."""
    n = case["n_fine"]
    f = torch.fft.irfftn(_field(g, n, -2.0, 0.5)[0], s=(n,) * 3)
    rho = torch.exp(1.2 * f / f.std()) + 0.04 * torch.rand((n, n, n), generator=g, device="cuda")
    if not case["tile"]:
        return None, rho
    return rho.reshape(n // R, R, n // R, R, n // R, R).sum((1, 3, 5)).contiguous(), rho


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = {"case": case, "pm": PM(_config(case))}
    pm, kind = s["pm"], case["kind"]
    if kind in ("step", "deposit", "pp"):
        s["codes"] = _codes(g, case)
    if kind == "step":
        s["b"] = [pm.empty_codes(c.n) for c in s["codes"]]
        s["c"] = [pm.empty_codes(c.n) for c in s["codes"]]
        if case["tuned"]:
            pm.set_tuning(TUNING)
        if case["graphs"]:
            pm.set_graphs(True)
    elif kind == "solve":
        s["rho"] = _densities(g, case)
        s["acc"] = pm.zeros_acc()
    elif kind in ("plain", "reverse", "restart"):
        s["x"], s["v"] = _particles(g, case)
        if kind == "reverse":
            s["lam"] = [[torch.randn(x.shape, generator=g, device="cuda") for x in s["x"]] for _ in range(2)]
    return s


def run(state):
    case, pm = state["case"], state["pm"]
    kind, ck, cd = case["kind"], case["c_kick"], case["c_drift"]
    if kind == "step":
        a, b, c = state["codes"], state["b"], state["c"]
        pm.step(a, b, ck, cd)
        pm.step(b, c, ck, cd)
        rho = pm.zeros_meshes()
        pm.deposit_codes(c, *rho)
        return {"rho_coarse": rho[0], "rho_fine": rho[1], "vmax": [c[0].vmax, c[1].vmax]}
    if kind == "solve":
        pm.solve(*state["rho"], *state["acc"])
        return {"acc_coarse": state["acc"][0], "acc_fine": state["acc"][1]}
    if kind == "deposit":
        rho = pm.zeros_meshes()
        pm.deposit_codes(state["codes"], *rho)
        return {"rho_coarse": rho[0], "rho_fine": rho[1]}
    if kind == "plain":
        x, v = [t.clone() for t in state["x"]], [t.clone() for t in state["v"]]
        acc = pm.step_plain(x, v, ck, cd, fixed=False)
        return {"x": x, "v": v, "acc_fine": acc}
    if kind == "reverse":
        x, v = [t.clone() for t in state["x"]], [t.clone() for t in state["v"]]
        lx, lv = ([t.clone() for t in lam] for lam in state["lam"])
        acc = pm.step_plain(x, v, ck, cd, fixed=True)
        pm.step_adjoint(state["x"], lx, lv, ck, cd, acc_fine=acc)
        return {"x": x, "v": v, "acc_fine": acc, "lam_x": lx, "lam_v": lv}
    if kind == "restart":
        out = {}
        for s, name in enumerate(("cdm", "nu")):
            codes = pm.compress(s, state["x"][s], state["v"][s])
            x, v = pm.decompress(s, codes)
            number = torch.zeros((pm.n_fine,) * 3, dtype=torch.int64, device="cuda")
            coarse = torch.zeros((pm.n_coarse,) * 3, dtype=torch.int64, device="cuda") if pm.two_level else None
            pm.deposit_fixed(s, x, coarse, number)
            out[name] = {"cnt": codes.cnt, "vmax": codes.vmax, "number_fine": number, "number_coarse": coarse,
                         "momentum": pm.deposit_weights(x, v)}
        return out
    return pm.pp_accel(state["codes"])


# ---- what a pass cannot do without -----------------------------------------

def work(case):
    n, kind = case["n_fine"], case["kind"]
    mesh, coarse = n ** 3, (n // R) ** 3 if case["tile"] else 0
    parts = case["n_cdm"] ** 3 + case["n_nu"] ** 3
    words = 4 + (8 if case["vel_bits"] == 16 else 4)         # codes of one particle in memory
    codes = parts * words + 2 * (n // R) ** 3

    def transform(edge):                                     # one forward and three inverse real transforms
        return 4 * 2.5 * edge ** 3 * math.log2(edge ** 3)

    if case["tile"]:
        solve = (n // case["tile"]) ** 3 * transform(case["tile"] + 2 * case["buffer"]) + transform(n // R)
    else:
        solve = transform(n)
    if kind == "step":       # codes read, written, read, written, read; the meshes written
        return {"bytes": 5 * codes + 4 * (mesh + coarse), "flops": 2 * solve + 250.0 * parts}
    if kind == "solve":
        return {"bytes": 16 * (mesh + coarse), "flops": solve}
    if kind == "deposit":
        return {"bytes": 4 * parts + 2 * (n // R) ** 3 + 4 * (mesh + coarse), "flops": 30.0 * parts}
    if kind == "plain":
        return {"bytes": 48 * parts + 12 * mesh, "flops": solve + 120.0 * parts}
    if kind == "reverse":
        return {"bytes": 96 * parts + 12 * mesh, "flops": 2 * solve + 300.0 * parts}
    if kind == "restart":
        return {"bytes": 24 * parts + 2 * (8 * (mesh + coarse) + 12 * mesh), "flops": 120.0 * parts}
    return {"bytes": 20 * parts, "flops": 30.0 * parts}


# ---- the same in 64 bits, by torch alone ------------------------------------

def _corners(x, n):
    """The 8 corners of periodic CIC: (mesh index, weight) of particles x (float64, mesh units)."""
    i0 = x.detach().floor()
    f = x - i0
    i0 = i0.long()
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                w = 1.0
                for d, up in ((0, dx), (1, dy), (2, dz)):
                    w = w * (f[:, d] if up else 1.0 - f[:, d])
                idx = ((i0[:, 2] + dz) % n * n + (i0[:, 1] + dy) % n) * n + (i0[:, 0] + dx) % n
                yield idx, w


def _cic(x, m, n):
    rho = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    for idx, w in _corners(x, n):
        rho = rho.index_add(0, idx, m * w)
    return rho.reshape(n, n, n)


def _gather(F, x, n):
    return sum(w[:, None] * F.reshape(3, -1)[:, idx].T for idx, w in _corners(x, n))


def _periodic(rho, h, r_s):
    """4 pi G i k exp(-k^2 r_s^2) rho(k) / k^2 on a periodic mesh of spacing h; k_d = 0 at the Nyquist index."""
    n = rho.shape[0]
    k = 2 * math.pi / (n * h) * torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    kg = torch.where(torch.arange(n, device="cuda") == n // 2, torch.zeros_like(k), k)
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + k[None, None, :n // 2 + 1] ** 2
    g = torch.where(k2 > 0, 4 * math.pi * G * torch.exp(-k2 * r_s * r_s) / k2.clamp_min(1e-300), torch.zeros_like(k2))
    dk = torch.fft.rfftn(rho) * (g / h ** 3)
    grad = (kg[None, None, :n // 2 + 1], kg[None, :, None], kg[:, None, None])
    return torch.stack([torch.fft.irfftn(1j * kd * dk, s=(n, n, n)) for kd in grad])


def _short_range(rho, r_s, cut):
    """Convolution with -G r S(r) / r^3, r <= cut: what every tile's interior holds."""
    n = rho.shape[0]
    m = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=torch.float64)
    r = (m[:, None, None] ** 2 + m[None, :, None] ** 2 + m[None, None, :] ** 2).sqrt()
    shape = torch.erfc(r / (2 * r_s)) + r / (r_s * math.sqrt(math.pi)) * torch.exp(-r * r / (4 * r_s * r_s))
    coef = torch.where((r > 0) & (r <= cut), -G * shape / r.clamp_min(0.5) ** 3, torch.zeros_like(r))
    rk = torch.fft.rfftn(rho)
    return torch.stack([torch.fft.irfftn(torch.fft.rfftn(coef * rd) * rk, s=(n, n, n))
                        for rd in (m[None, None, :], m[None, :, None], m[:, None, None])])


def _accelerations(case, rho_coarse, rho_fine):
    if not case["tile"]:
        return None, _periodic(rho_fine, 1.0, 0.0)
    cut = _r_cut(case)
    return _periodic(rho_coarse, float(R), cut / 4.5), _short_range(rho_fine, cut / 4.5, cut)


def _decoded(codes, n_cmp):
    """Positions of the particles of one species' codes (bin centres)."""
    count = codes.cnt.long()
    k = int(codes.n_esc)
    count[codes.esc[:k, 0].long()] = codes.esc[:k, 1].long()
    cell = torch.repeat_interleave(torch.arange(n_cmp ** 3, device="cuda"), count)
    c = torch.stack([cell % n_cmp, (cell // n_cmp) % n_cmp, cell // (n_cmp * n_cmp)], dim=1).double()
    return (c + (codes.pos[:, :3].double() + 0.5) / 256.0) * R


def _both_meshes(case, xs):
    n = case["n_fine"]
    fine = sum(_cic(x, MASS[s], n) for s, x in enumerate(xs))
    coarse = sum(_cic(x / R, MASS[s], n // R) for s, x in enumerate(xs)) if case["tile"] else None
    return coarse, fine


def _step64(case, x, v):
    n = case["n_fine"]
    coarse, fine = _accelerations(case, *_both_meshes(case, x))
    out_x, out_v = [], []
    for xs, vs in zip(x, v):
        a = _gather(fine, xs, n)
        if coarse is not None:
            a = a + _gather(coarse, xs / R, n // R)
        out_v.append(vs + case["c_kick"] * a)
        out_x.append(xs + case["c_drift"] * out_v[-1])
    return out_x, out_v, fine


def _wrap64(x, n):
    """x in the box: a position that float32 rounds onto the far face belongs to the near one."""
    return x - n * torch.floor(x.float() / n).double()


def exact(case, seed):
    kind, n = case["kind"], case["n_fine"]
    s = prepare(case, seed) if kind != "step" else None
    if kind == "solve":
        rho = [None if r is None else r.double() for r in s["rho"]]
        coarse, fine = _accelerations(case, *rho)
        return {"acc_coarse": coarse, "acc_fine": fine}
    if kind == "deposit":
        coarse, fine = _both_meshes(case, [_decoded(c, n // R) for c in s["codes"]])
        return {"rho_coarse": coarse, "rho_fine": fine}
    if kind == "plain":
        x, v, fine = _step64(case, [t.double() for t in s["x"]], [t.double() for t in s["v"]])
        return {"x": [_wrap64(t, n) for t in x], "v": v, "acc_fine": fine}
    if kind == "reverse":
        x0 = [t.double().requires_grad_() for t in s["x"]]
        v0 = [t.double().requires_grad_() for t in s["v"]]
        x, v, fine = _step64(case, x0, v0)
        lam = [t.double() for t in s["lam"][0] + s["lam"][1]]
        grad = torch.autograd.grad(x + v, x0 + v0, lam)
        return {"x": [_wrap64(t.detach(), n) for t in x], "v": [t.detach() for t in v],
                "acc_fine": fine.detach(), "lam_x": list(grad[:2]), "lam_v": list(grad[2:])}
    if kind == "restart":
        out = {}
        half = 1 << (case["vel_bits"] - 1)
        for k, name in enumerate(("cdm", "nu")):
            x, v = s["x"][k], s["v"][k]
            u = x / R
            c = u.floor()
            x = (c.double() + (torch.floor((u - c) * 256).clamp(max=255).double() + 0.5) / 256) * R
            vmax = v.abs().max()
            q = torch.floor(v * (half / vmax) + half).clamp(0, 2 * half - 1)
            v = ((q.double() - half) + 0.5) * (vmax.double() / half)
            momentum = torch.stack([_cic(x, v[:, d], n) for d in range(3)])
            out[name] = {"cnt": None, "vmax": vmax.double().reshape(1), "number_fine": None, "number_coarse": None,
                         "momentum": momentum}
        return out
    if kind == "pp":
        r_soft = n / (20.0 * case["n_cdm"])
        x = torch.cat([_decoded(c, n // R) for c in s["codes"]])
        m = torch.cat([torch.full((c.n,), MASS[k], dtype=torch.float64, device="cuda")
                       for k, c in enumerate(s["codes"])])
        f = x.floor().long()
        cell, order = torch.sort(f[:, 0] + n * (f[:, 1] + n * f[:, 2]))
        xs, ms = x[order], m[order]
        acc = torch.zeros((x.shape[0], 4), dtype=torch.float64, device="cuda")
        for k in range(1, int(torch.bincount(cell).max())):
            same = torch.nonzero(cell[k:] == cell[:-k]).reshape(-1)
            d = xs[same + k] - xs[same]
            r2 = d.square().sum(1)
            w = torch.where(r2 >= r_soft * r_soft, G / r2.clamp_min(1e-12) ** 1.5, torch.zeros_like(r2))[:, None]
            acc[:, :3].index_add_(0, same, w * d * ms[same + k][:, None])
            acc[:, :3].index_add_(0, same + k, -w * d * ms[same][:, None])
        out = torch.empty_like(acc)
        out[order] = acc
        return out
    return None
