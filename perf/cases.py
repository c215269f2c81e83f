"""The work a user of this framework has it do, as cases that can be timed.

Families (the "family" of a case):
  star     synchronised steps of the production mesh: a stretched polytrope by a
           point mass with excision, PPM, tabulated EOS, dual energy
  wave     synchronised steps of a cold advected entropy wave: PLM, tabulated EOS, dual
           energy, periodic
  gas      synchronised steps of a smooth ideal-gas flow: PPM, outflow, blocks of uneven
           sizes
  lat      one window of localized adaptive time stepping of a thin stream
  eos      (rho, e) -> T, P, cs^2 of an array of cells
  gravity  a self-gravity solve from the full-multigrid start
  remap    a state onto another mesh
  train    training of the learned EOS guess
Every case goes through the public Python binding on the current CUDA stream.
"""
import os

import numpy as np
import torch

from paper_2609_37859_gb300 import tde
from paper_2609_37859_gb300 import workloads as wl

TABLE = os.path.join(os.path.dirname(os.path.abspath(wl.__file__)), "data", "eos_saha_hhe_256.npz")
CFL = 0.3
G_CODE = wl.G_CODE
STAR_FLOORS = (1e-8, 1e-10)      # density and pressure floors of the star's mesh (code units)
WAVE = dict(rho0=1e-8, T0=1e3, mach=1e7, amp=1e-3, floor=1e-20)
DEV = "cuda:0"

_kept = {}


def _context():
    if "ctx" not in _kept:
        _kept["ctx"] = tde.Context(0)
    return _kept["ctx"]


def _eos(learned=False):
    """The table on the device, and (learned) with its network trained: a program
    loads and trains once and keeps the handle."""
    if "eos" not in _kept:
        _kept["eos"] = tde.EOS.from_file(_context(), TABLE)
    if learned and "net" not in _kept:
        _kept["net"] = _kept["eos"].train(seed=2609, n_samples=1 << 20, epochs=20, batch=4096, lr=3e-3)
    return _kept["eos"]


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest mesh in use (the smoke check's and the tests'): a step is a few
        # dozen microseconds of launches
        {"name": "step_wave_32", "family": "wave", "nx": 32, "ny": 32, "nz": 32, "block": 16},
        # the benchmark's entropy wave, 64 MeshBlocks of 32^3
        {"name": "step_wave_128", "family": "wave", "nx": 128, "ny": 128, "nz": 128, "block": 32},
        # uneven blocks (odd widths, remainders), ideal gas, the production run's HLLE solver
        {"name": "step_gas_ragged", "family": "gas", "nx": 85, "ny": 63, "nz": 45, "block": 24, "hlle": True,
         "dual": False},
        # the production-shaped mesh around the star with the learned closure: the
        # benchmark's cells and scheme, 256 of its MeshBlocks
        {"name": "step_star_8m", "family": "star", "bx": 8, "by": 8, "bz": 4, "block": 32, "learned": True,
         "hlle": False},
        # one window of the stream workload (table bisection, replayed as a CUDA graph): the
        # benchmark's 512 MeshBlocks and time-step levels, with 16^3 cells in a block
        {"name": "lat_stream", "family": "lat", "rx": 10, "ry": 10, "rz": 4, "block": 16, "split": 16, "n_lat": 5},
        # EOS calls: a handful of cells (an initial condition's profile), the benchmark's
        # batch, and the learned form on an odd count
        {"name": "eos_5k", "family": "eos", "n": 5001, "mode": "bisect"},
        {"name": "eos_16m", "family": "eos", "n": 1 << 24, "mode": "bisect"},
        {"name": "eos_learned_6m", "family": "eos", "n": 6_000_001, "mode": "learned"},
        # self-gravity: the benchmark's periodic grid, and a smaller isolated cloud with
        # multipole boundary values
        {"name": "gravity_256", "family": "gravity", "nb": 8, "nbz": 8, "block": 32, "isolated": False},
        {"name": "gravity_iso_64", "family": "gravity", "nb": 4, "nbz": 4, "block": 16, "isolated": True},
        # a remap onto a grid twice as fine (half the domain along z)
        {"name": "remap_refine_128", "family": "remap", "n": 128, "block": 32, "refine": True},
        # training of the learned guess: two epochs of the usual batch
        {"name": "train_guess", "family": "train", "samples": 1 << 18, "epochs": 2, "batch": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    f = rng.choice(["star", "wave", "gas", "lat", "eos", "eos", "gravity", "remap", "train"])
    if f == "star":
        return {"family": f, "bx": rng.randint(2, 7), "by": rng.randint(2, 6), "bz": rng.randint(1, 4), "block": rng.choice([16, 20, 32]),
                "learned": rng.random() < 0.5, "hlle": rng.random() < 0.5}
    if f == "wave":
        return {"family": f, "nx": _log_int(rng, 24, 128), "ny": _log_int(rng, 16, 128), "nz": _log_int(rng, 16, 128),
                "block": rng.choice([16, 24, 32])}
    if f == "gas":
        return {"family": f, "nx": _log_int(rng, 20, 180), "ny": _log_int(rng, 20, 150), "nz": _log_int(rng, 20, 120),
                "block": rng.choice([15, 16, 24, 32]), "hlle": rng.random() < 0.5, "dual": rng.random() < 0.5}
    if f == "lat":
        b = rng.choice([16, 32])
        m = 1 if b == 32 else 2
        return {"family": f, "rx": m * rng.randint(4, 5), "ry": m * rng.randint(4, 5), "rz": m * rng.randint(1, 2),
                "block": b, "split": m * rng.randint(2, 4), "n_lat": rng.randint(3, 5)}
    if f == "eos":
        return {"family": f, "n": _log_int(rng, 1000, 1 << 24), "mode": rng.choice(["bisect", "learned", "plain"])}
    if f == "gravity":
        nb = rng.choice([1, 2, 4])   # (the solver takes power-of-two directions)
        return {"family": f, "nb": nb, "nbz": rng.choice([nb, 2 * nb]), "block": rng.choice([16, 32, 64]),
                "isolated": rng.random() < 0.5}
    if f == "remap":
        return {"family": f, "n": rng.choice([48, 64, 80, 96, 128]), "block": rng.choice([16, 32]), "refine": rng.random() < 0.5}
    return {"family": f, "samples": 4096 * rng.randint(8, 64), "epochs": rng.randint(1, 3), "batch": rng.choice([2048, 4096, 8192])}


# ------------------------------------------------------------------ inputs

def _centres(lay):
    ax = [lay.xmin[a] + (torch.arange(lay.N[a], dtype=torch.float64, device=DEV) + 0.5) * lay.dx[a] for a in range(3)]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _smooth(lay, gen, amp, modes):
    """A sum of low Fourier modes on the global grid [Nz, Ny, Nx]."""
    x, y, z = _centres(lay)
    L = [lay.dx[a] * lay.N[a] for a in range(3)]
    f = torch.zeros((lay.N[2], lay.N[1], lay.N[0]), dtype=torch.float64, device=DEV)
    for _ in range(modes):
        k = torch.randint(0, 3, (3,), generator=gen).tolist()
        ph = float(torch.rand(1, generator=gen, dtype=torch.float64)) * 2 * np.pi
        f += torch.sin(2 * np.pi * (k[0] * x / L[0] + k[1] * y / L[1] + k[2] * z / L[2]) + ph)
    return amp * f / modes


def _smooth_prims(lay, seed, drho, dv, dP, modes):
    gen = torch.Generator().manual_seed(int(seed))
    r = 1.0 + _smooth(lay, gen, drho, modes)
    v = [_smooth(lay, gen, dv, modes) for _ in range(3)]
    return torch.stack([r, *v, 1.0 + _smooth(lay, gen, dP, modes)])


def _pack(lay, G):
    """Global [n, Nz, Ny, Nx] -> the MeshBlock layout [n, ntot] (ghost cells zero)."""
    U = torch.zeros((G.shape[0], lay.ntot), dtype=torch.float64, device=DEV)
    gx, gy, gz = lay.gofs(0), lay.gofs(1), lay.gofs(2)
    for b in range(lay.nb):
        i0, j0, k0, nx, ny, nz = (int(q) for q in lay.blocks[b])
        px, py, pz = (int(q) for q in lay.pd[b])
        V = U[:, int(lay.off[b]):int(lay.off[b + 1])].view(-1, pz, py, px)
        V[:, gz:gz + nz, gy:gy + ny, gx:gx + nx] = G[:, k0:k0 + nz, j0:j0 + ny, i0:i0 + nx]
    return U


def _table():
    if "table" not in _kept:
        d = np.load(TABLE)
        t = {k: torch.tensor(np.asarray(d[k], dtype=np.float64), device=DEV) for k in ("log10_e", "log10_P", "log10_cs2")}
        t["nr"], t["nt"] = int(d["n_rho"]), int(d["n_T"])
        t["lr"], t["lT"] = tuple(float(q) for q in d["lrho"]), tuple(float(q) for q in d["lT"])
        for k in ("log10_e", "log10_P", "log10_cs2"):
            t[k] = t[k].reshape(t["nr"], t["nt"])
        _kept["table"] = t
    return _kept["table"]


def _wave_setup(case, seed):
    N, b = (case["nx"], case["ny"], case["nz"]), case["block"]
    lay = wl.uniform_layout(N, (b, b, b), bc=(1, 1, 1), ng=2)
    r, T = (torch.tensor([WAVE[k]], dtype=torch.float64, device=DEV) for k in ("rho0", "T0"))
    Pw, cs2 = _x_eval_rhoT(r, T)
    phi = 2 * np.pi * float(torch.rand(1, generator=torch.Generator().manual_seed(int(seed)), dtype=torch.float64))
    x = _centres(lay)[0]
    one = torch.ones((N[2], N[1], N[0]), dtype=torch.float64, device=DEV)
    rho = WAVE["rho0"] * (1 + WAVE["amp"] * torch.sin(2 * np.pi * x + phi)) * one
    W = torch.stack([rho, one * (WAVE["mach"] * float(cs2) ** 0.5), 0 * one, 0 * one, one * float(Pw)])
    f = WAVE["floor"]
    par = dict(eos=tde.EOS_TABLE, dual=1, eta1=1e-3, eta2=1e-4, rho_floor=f, p_floor=f, u_floor=f)
    return lay, W, par, None


def _gas_setup(case, seed):
    N, b = (case["nx"], case["ny"], case["nz"]), case["block"]
    lay = wl.uniform_layout(N, (b, b - 3, b - 7), bc=(0, 0, 0), ng=3)
    W = _smooth_prims(lay, seed, 0.4, 0.6, 0.4, 4)
    par = dict(recon=tde.RECON_PPM, dual=int(case["dual"]), eta1=1e-3, eta2=1e-4, rho_floor=1e-12, p_floor=1e-12,
               u_floor=1e-12, riemann=tde.RIEMANN_HLLE if case["hlle"] else tde.RIEMANN_HLLC)
    return lay, W, par, None


def _star_setup(case, seed):
    nb, b = (case["bx"], case["by"], case["bz"]), case["block"]
    half = tuple(n * b * 0.0625 / 2.0 for n in nb)   # Rsun: cells of 1/16 Rsun
    # the point mass is inside the mesh, off the star (and off the cells' symmetry points,
    # where a cell could lie exactly on the excision sphere)
    at = (0.5471 * half[0], 0.4473 * half[1], 0.0131 * half[2])
    lay, f, b_ = wl.star_c5(seed=seed, rho_floor=STAR_FLOORS[0], p_floor=STAR_FLOORS[1], n_blocks=nb, block=b,
                            half_rsun=half, bh_at_rsun=at, stretch=4.0)
    W = torch.stack([torch.from_numpy(np.ascontiguousarray(f[k])).to(DEV) for k in ("rho", "vx", "vy", "vz", "P")])
    par = dict(eos=tde.EOS_TABLE, recon=tde.RECON_PPM, dual=1, eta1=1e-3, eta2=1e-4, rho_floor=STAR_FLOORS[0],
               p_floor=STAR_FLOORS[1], u_floor=1.5 * STAR_FLOORS[1], unit_rho=wl.RHO0_CGS, unit_e=wl.V0_CGS ** 2,
               eos_mode=tde.INVERT_SURROGATE if case["learned"] else tde.INVERT_BISECT,
               riemann=tde.RIEMANN_HLLE if case["hlle"] else tde.RIEMANN_HLLC)
    # (held at its place: every pass steps from the same state and would otherwise move it on)
    bh = dict(on=1, excise=1, GM=b_["GM"], r_soft=b_["r_soft"], r_exc=b_["r_exc"], x0=b_["x0"])
    return lay, W, par, bh


STEPS = {"wave": _wave_setup, "gas": _gas_setup, "star": _star_setup}


def _lat_setup(case, seed):
    u = torch.rand(4, generator=torch.Generator().manual_seed(int(seed)), dtype=torch.float64).tolist()
    lay, f, b = wl.stream_c4(split_nearest=case["split"], n_root=(case["rx"], case["ry"], case["rz"]), block=case["block"],
                             sigma_rsun=0.9 + 0.4 * u[0], rp_rsun=9.5 + u[1], ra_rsun=27.0 + u[2],
                             rho_peri=10.0 ** (-2.0 + 0.2 * u[3]))
    rho = torch.from_numpy(np.ascontiguousarray(f["rho"])).to(DEV)
    P, _ = _x_eval_rhoT((rho * wl.RHO0_CGS).reshape(-1), torch.from_numpy(np.ascontiguousarray(f["T"])).to(DEV).reshape(-1))
    P = P.reshape(rho.shape) / (wl.RHO0_CGS * wl.V0_CGS ** 2)
    W = torch.stack([rho, *(torch.from_numpy(np.ascontiguousarray(f[k])).to(DEV) for k in ("vx", "vy", "vz")), P])
    par = dict(eos=tde.EOS_TABLE, recon=tde.RECON_PPM, dual=1, eta1=1e-3, eta2=1e-4, rho_floor=1e-17, p_floor=1e-30,
               u_floor=1.5e-30, unit_rho=wl.RHO0_CGS, unit_e=wl.V0_CGS ** 2)
    bh = dict(on=1, excise=1, GM=b["GM"], r_soft=b["r_soft"], r_exc=b["r_exc"], x0=b["x0"])
    return lay, W, par, bh


def _eos_inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    rho, T = wl.c3_inputs(case["n"], gen, DEV)
    return rho, _x_eval(rho, T, "log10_e")


def _gravity_setup(case, seed):
    n, nz = case["nb"] * case["block"], case["nbz"] * case["block"]
    bc, h = (0, 0, 0) if case["isolated"] else (1, 1, 1), nz / n
    lay = wl.uniform_layout((n, n, nz), (case["block"],) * 3, domain=((-1, 1), (-1, 1), (-h, h)), bc=bc, ng=2)
    W = _smooth_prims(lay, seed, 0.5, 0.1, 0.2, 4)
    if case["isolated"]:   # a centrally condensed cloud over a thin floor
        x, y, z = _centres(lay)
        s = 0.05 * (W[0, 0, 0, 0] - 1.0)
        W[0] = 1e-4 + W[0] * torch.exp(-((x - 0.1 - s) ** 2 + y ** 2 + (z + 0.05) ** 2) / (2 * 0.2 ** 2))
        W[4] = 0.1 * W[0]
    return lay, W


def _remap_setup(case, seed):
    n, b = case["n"], (case["block"],) * 3
    src = wl.uniform_layout((n, n, n), b, ((-1, 1),) * 3, bc=(0, 0, 0), ng=2)
    if case["refine"]:
        dst = wl.uniform_layout((2 * n, 2 * n, n), b, ((-1, 1), (-1, 1), (-0.5, 0.5)), bc=(0, 0, 0), ng=2)
    else:
        dst = wl.uniform_layout((n, n, n), b, ((-2, 2),) * 3, bc=(0, 0, 0), ng=2)
    return src, dst, _smooth_prims(src, seed, 0.5, 0.3, 0.2, 4)


def prepare(case, seed):
    ctx, f = _context(), case["family"]
    if f in STEPS:
        lay, W, par, bh = STEPS[f](case, seed)
        eos = _eos(bool(case.get("learned"))) if par.get("eos") else None
        mesh = tde.Mesh(ctx, lay, tde.make_params(**par), eos)
        mesh.prim_to_cons(_pack(lay, W))
        return {"run": _run_step, "mesh": mesh, "U0": mesh.U.clone(), "bh": tde.make_bh(**bh) if bh else None,
                "dt": torch.zeros(1, dtype=torch.float64, device=DEV)}
    if f == "lat":
        lay, W, par, bh = _lat_setup(case, seed)
        mesh = tde.Mesh(ctx, lay, tde.make_params(**par), _eos())
        mesh.prim_to_cons(_pack(lay, W))
        b = tde.make_bh(**bh)
        mesh.lat_assign(case["n_lat"], CFL, merge_frac=0.01, bh=b)
        return {"run": _run_lat, "mesh": mesh, "U0": mesh.U.clone(), "bh": b}
    if f == "eos":
        eos = _eos(case["mode"] == "learned")
        rho, e = _eos_inputs(case, seed)
        mode = {"bisect": tde.INVERT_BISECT, "learned": tde.INVERT_SURROGATE, "plain": tde.INVERT_BISECT_PLAIN}[case["mode"]]
        return {"run": _run_eos, "eos": eos, "rho": rho, "e": e, "mode": mode, "out": [torch.empty_like(rho) for _ in range(3)]}
    if f == "gravity":
        lay, W = _gravity_setup(case, seed)
        mesh = tde.Mesh(ctx, lay, tde.make_params())
        mesh.prim_to_cons(_pack(lay, W))
        return {"run": _run_gravity, "mesh": mesh, "isolated": case["isolated"]}
    if f == "remap":
        src, dst, W = _remap_setup(case, seed)
        a = tde.Mesh(ctx, src, tde.make_params(dual=1))
        a.prim_to_cons(_pack(src, W))
        return {"run": _run_remap, "src": a, "dst": tde.Mesh(ctx, dst, tde.make_params(dual=1, rho_floor=1e-8, u_floor=1e-10))}
    return {"run": _run_train, "eos": tde.EOS.from_file(ctx, TABLE), "seed": int(seed),
            "case": {k: case[k] for k in ("samples", "epochs", "batch")}}


# ------------------------------------------------------------------ the passes

def run(state):
    return state["run"](state)


def _run_step(s):
    # one synchronised step from the state in hand (a copy on the device, so that every
    # pass does the same step)
    m = s["mesh"]
    m.U.copy_(s["U0"])
    m.step(cfl=CFL, bh=s["bh"], dt_out=s["dt"])
    return {"U": m.U, "dt": s["dt"]}


def _run_lat(s):
    m = s["mesh"]
    m.U.copy_(s["U0"])
    updates = m.lat_window(bh=s["bh"], use_graph=True)
    return {"U": m.U, "updates": updates}


def _run_eos(s):
    T, P, c2 = s["out"]
    s["eos"].invert(s["rho"], s["e"], T=T, P=P, cs2=c2, mode=s["mode"])
    return {"T": T, "P": P, "cs2": c2}


def _run_gravity(s):
    m = s["mesh"]
    cycles, _ = m.gravity_solve(G_CODE, 0.0, tol=1e-9, max_cycles=30, warm=False, isolated=s["isolated"], lmax=4, fmg=True)
    return {"phi": m.gravity_phi(), "cycles": cycles}


def _run_remap(s):
    return {"U": s["dst"].remap_from(s["src"], s["src"].U)}


def _run_train(s):
    # from the seeded initial weights, as a program's first training is
    c = s["case"]
    s["eos"].reset_weights_for_training()
    r = s["eos"].train(seed=s["seed"], n_samples=c["samples"], epochs=c["epochs"], batch=c["batch"], lr=3e-3)
    return {"weights": s["eos"].get_weights(), "loss_last": np.float32(r["loss_last"])}


def work(case):
    f = case["family"]
    if f in STEPS or f == "lat":
        if f == "star":
            n = case["bx"] * case["by"] * case["bz"] * case["block"] ** 3
        elif f == "lat":   # about a quarter of the blocks in each of up to 2^n_lat fine steps
            n = case["rx"] * case["ry"] * case["rz"] * case["block"] ** 3
            n = n * 2 ** case["n_lat"] // 4 if case["block"] < 32 else 2 * n
        else:
            n = case["nx"] * case["ny"] * case["nz"]
        nvar = 5 if f == "gas" and not case["dual"] else 6
        # a stage reads and writes the state, the second also the step's start; FP64
        # operations of two stages: conversion, three sweeps (reconstruction, Riemann
        # solve, divergence), sources and update
        per = {"wave": 2 * 800, "gas": 2 * 620, "star": 2 * 950, "lat": 2 * 950}[f]
        return {"bytes": 5 * nvar * 8 * n, "flops": per * n}
    if f == "eos":   # two numbers in, three out; two logarithms, three exponentials, the lookups
        return {"bytes": 40 * case["n"], "flops": 150 * case["n"]}
    if f == "gravity":   # density in, potential out; a full-multigrid start and four V-cycles
        n = case["nb"] ** 2 * case["nbz"] * case["block"] ** 3
        return {"bytes": 16 * n, "flops": 5 * 100 * n}
    if f == "remap":
        n = case["n"] ** 3
        dst = 4 * n if case["refine"] else n
        return {"bytes": 48 * ((n // 2 if case["refine"] else n) + dst), "flops": 100 * dst}
    n = case["samples"] * case["epochs"]   # 4482 weights, forward and backward
    return {"bytes": 16 * case["samples"] + 4482 * 4, "flops": 6 * 4482 * n}


# ------------------------------------------------- the same in plain torch, 64 bits

def _x_cell(t, x, n):
    i = torch.clamp(torch.floor(x), 0, n - 2).long()
    return i, x - i


def _x_bilin(t, f, i, w, j, s):
    F = t[f]
    lo = (1 - s) * F[i, j] + s * F[i, j + 1]
    hi = (1 - s) * F[i + 1, j] + s * F[i + 1, j + 1]
    return (1 - w) * lo + w * hi


def _x_rho(t, rho):
    x = (torch.log10(rho) - t["lr"][0]) * ((t["nr"] - 1) / (t["lr"][1] - t["lr"][0]))
    cl = ~((x >= 0) & (x <= t["nr"] - 1))
    i, w = _x_cell(t, torch.clamp(torch.nan_to_num(x, nan=0.0), 0, t["nr"] - 1), t["nr"])
    return i, w, cl


def _x_eval(rho, T, *names):
    t = _table()
    i, w, _ = _x_rho(t, rho)
    y = torch.clamp((torch.log10(T) - t["lT"][0]) * ((t["nt"] - 1) / (t["lT"][1] - t["lT"][0])), 0, t["nt"] - 1)
    j, s = _x_cell(t, y, t["nt"])
    out = [10.0 ** _x_bilin(t, n, i, w, j, s) for n in names]
    return out[0] if len(out) == 1 else out


def _x_eval_rhoT(rho, T):
    return _x_eval(rho, T, "log10_P", "log10_cs2")


def _x_invert(rho, e):
    """T, P, cs2, the energy the table represents, clamped?"""
    t = _table()
    i, w, cl = _x_rho(t, rho)
    E, nt = t["log10_e"], t["nt"]
    y = torch.where(e > 0, torch.log10(torch.clamp(e, min=1e-300)), torch.full_like(e, -float("inf")))

    def g(j):
        return (1 - w) * E[i, j] + w * E[i + 1, j]
    lo, hi = torch.zeros_like(i), torch.full_like(i, nt - 1)
    while bool(((hi - lo) > 1).any()):
        mid = (lo + hi) // 2
        below = g(mid) <= y
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, torch.maximum(mid, lo + 1))
    j = torch.clamp(lo, max=nt - 2)
    s = (y - g(j)) / (g(j + 1) - g(j))
    cold, hot = y <= g(torch.zeros_like(i)), y >= g(torch.full_like(i, nt - 1))
    j = torch.where(cold, torch.zeros_like(j), torch.where(hot, torch.full_like(j, nt - 2), j))
    s = torch.where(cold, torch.zeros_like(s), torch.where(hot, torch.ones_like(s), s))
    cl = cl | cold | hot
    dlt = (t["lT"][1] - t["lT"][0]) / (nt - 1)
    T = 10.0 ** (t["lT"][0] + (j + s) * dlt)
    P, c2, eu = (10.0 ** _x_bilin(t, n, i, w, j, s) for n in ("log10_P", "log10_cs2", "log10_e"))
    return T, P, c2, torch.where(cl, eu, e), cl


def _x_energy_of_P(rho, P):
    """Specific internal energy at (rho, P), cgs."""
    t = _table()
    i, w, _ = _x_rho(t, rho)
    lp = torch.log10(P)
    lo, hi = torch.zeros_like(lp), torch.full_like(lp, float(t["nt"] - 1))
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        j, s = _x_cell(t, mid, t["nt"])
        below = _x_bilin(t, "log10_P", i, w, j, s) < lp
        lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
    j, s = _x_cell(t, 0.5 * (lo + hi), t["nt"])
    return 10.0 ** _x_bilin(t, "log10_e", i, w, j, s)


class _Params:
    def __init__(self, par):
        d = dict(eos=0, recon=0, dual=0, gamma=5.0 / 3.0, eta1=1e-3, eta2=1e-4, rho_floor=1e-300, p_floor=1e-300,
                 u_floor=1e-300, unit_rho=1.0, unit_e=1.0, riemann=0)
        d.update({k: v for k, v in par.items() if k in d})
        self.__dict__.update(d)


def _x_p2c(p, W):
    r, vx, vy, vz, P = W
    if p.eos:
        U = r * (_x_energy_of_P((r * p.unit_rho).reshape(-1), (P * p.unit_rho * p.unit_e).reshape(-1)).reshape(r.shape) / p.unit_e)
    else:
        U = P / (p.gamma - 1)
    E = U + 0.5 * r * (vx * vx + vy * vy + vz * vz)
    return torch.stack([r, r * vx, r * vy, r * vz, E] + ([U] if p.dual else []))


def _x_closure(p, rho, U):
    """P, cs2, the represented U (code units)."""
    if not p.eos:
        P = (p.gamma - 1) * U
        return P, p.gamma * P / rho, U
    sh = rho.shape
    _, P, c2, eu, cl = (q.reshape(sh) for q in _x_invert((rho * p.unit_rho).reshape(-1), (U / rho * p.unit_e).reshape(-1)))
    return P / (p.unit_rho * p.unit_e), c2 / p.unit_e, torch.where(cl, rho * (eu / p.unit_e), U)


def _x_c2p(p, U):
    rho = torch.clamp(U[0], min=p.rho_floor)
    v = [U[1 + a] / rho for a in range(3)]
    Uc = U[4] - 0.5 * (U[1] * v[0] + U[2] * v[1] + U[3] * v[2])
    if p.dual:
        Uc = torch.where((Uc > 0) & (Uc > p.eta1 * U[4]), Uc, U[5])
    P, c2, Uu = _x_closure(p, rho, Uc)
    P = torch.clamp(P, min=p.p_floor)
    W = [rho, *v, P]
    if p.eos:
        W += [1.0 + P / Uu, rho * c2 / P]
    if p.dual:
        W.append(U[5])
    return W


def _x_pad(A, lay, d, n):
    """n ghost cells along direction d (0 = x), by the boundary."""
    k = A.dim() - 1 - d
    N = A.shape[k]
    idx = torch.arange(-n, N + n, device=A.device)
    idx = idx % N if lay.bc[d] == 1 else torch.clamp(idx, 0, N - 1)
    return A.index_select(k, idx)


def _x_sl(A, d, lo, hi):
    k = A.dim() - 1 - d
    return A.narrow(k, lo, A.shape[k] + hi - lo)


def _x_faces(p, q, d):
    """Low and high face values of cells -1 .. N from q padded by 3 cells."""
    if not p.recon:
        qm, q0, qp = _x_sl(q, d, 1, -3), _x_sl(q, d, 2, -2), _x_sl(q, d, 3, -1)
        dl, dr = q0 - qm, qp - q0
        pr = dl * dr
        h = torch.where(pr > 0, pr / torch.where(pr > 0, dl + dr, torch.ones_like(dl)), torch.zeros_like(dl))
        return q0 - h, q0 + h
    a, b, c, e = (_x_sl(q, d, k, k - 3) for k in range(4))
    f = (7.0 / 12.0) * (b + c) - (1.0 / 12.0) * (a + e)
    f = torch.minimum(torch.maximum(f, torch.minimum(b, c)), torch.maximum(b, c))
    aL, aR, q0 = _x_sl(f, d, 0, -1), _x_sl(f, d, 1, 0), _x_sl(q, d, 2, -2)
    flat = (aR - q0) * (q0 - aL) <= 0
    da, q6 = aR - aL, 6 * (q0 - 0.5 * (aL + aR))
    L = torch.where(da * da < da * q6, 3 * q0 - 2 * aR, aL)
    R = torch.where(da * q6 < -da * da, 3 * q0 - 2 * aL, aR)
    return torch.where(flat, q0, L), torch.where(flat, q0, R)


def _x_riemann(p, d, L, R):
    """Fluxes [5 or 6] and the face velocity from the face states' lists."""
    tbl = bool(p.eos)
    g = p.gamma

    def st(S):
        ge, g1 = (S[5], S[6]) if tbl else (g, g)
        U = S[4] / (ge - 1)
        E = U + 0.5 * S[0] * (S[1] ** 2 + S[2] ** 2 + S[3] ** 2)
        return S[1 + d], torch.sqrt(g1 * S[4] / S[0]), E
    ul, cl, El = st(L)
    ur, cr, Er = st(R)
    SL, SR = torch.minimum(ul - cl, ur - cr), torch.maximum(ul + cl, ur + cr)

    def cons(S, E):
        return [S[0], S[0] * S[1], S[0] * S[2], S[0] * S[3], E]

    def flux(S, u, E):
        m = S[0] * u
        F = [m, m * S[1], m * S[2], m * S[3], (E + S[4]) * u]
        F[1 + d] = F[1 + d] + S[4]
        return F
    UL, UR, FL, FR = cons(L, El), cons(R, Er), flux(L, ul, El), flux(R, ur, Er)
    if p.riemann == 1:
        bm, bp = torch.clamp(SL, max=0.0), torch.clamp(SR, min=0.0)
        den = bp - bm
        den = torch.where(den == 0, torch.ones_like(den), den)
        F = [(bp * a - bm * b + bp * bm * (v - u)) / den for a, b, u, v in zip(FL, FR, UL, UR)]
    else:
        al, ar = L[0] * (SL - ul), R[0] * (SR - ur)
        SM = (R[4] - L[4] + al * ul - ar * ur) / (al - ar)

        def star(S, u, E, Sk):
            den = Sk - SM
            den = torch.where(den == 0, torch.ones_like(den), den)
            r = S[0] * (Sk - u) / den
            V = [r, r * S[1], r * S[2], r * S[3], None]
            V[1 + d] = r * SM
            V[4] = E + (SM - u) * (E + S[4] + S[0] * (Sk - u) * SM) / den
            return V
        VL, VR = star(L, ul, El, SL), star(R, ur, Er, SR)
        F = []
        for q in range(5):
            sl = FL[q] + SL * (VL[q] - UL[q])
            sr = FR[q] + SR * (VR[q] - UR[q])
            F.append(torch.where(SL >= 0, FL[q], torch.where(SR <= 0, FR[q], torch.where(SM >= 0, sl, sr))))
    vf = None
    if p.dual:
        m = F[0]
        r = torch.where(m > 0, L[0], R[0])
        A = torch.where(m > 0, L[-1], R[-1])
        vf = m / r
        F.append(A * vf)
    return F, vf


class _BH:
    def __init__(self, lay, bh, t):
        r = [bh["x0"][a] + bh.get("v0", (0, 0, 0))[a] * t for a in range(3)]
        self.lay, self.bh, self.r = lay, bh, r

    def r2(self, d=None):
        """Squared distance on the grid, with one ghost cell along direction d."""
        s = 0.0
        for a in range(3):
            n = self.lay.N[a]
            i = torch.arange(-1, n + 1, device=DEV) if a == d else torch.arange(n, device=DEV)
            x = self.lay.xmin[a] + (i.double() + 0.5) * self.lay.dx[a] - self.r[a]
            s = s + (x * x).reshape([-1 if b == a else 1 for b in (2, 1, 0)])
        return s

    def phi(self, d):
        return -self.bh["GM"] / torch.sqrt(self.r2(d) + self.bh["r_soft"] ** 2)

    def inside(self, d=None):
        return torch.sqrt(self.r2(d)) < self.bh["r_exc"]


def _x_stage(p, lay, bh, stage, U0, Uin, dt, t):
    W = _x_c2p(p, Uin)
    nvar = 5 + p.dual
    acc, dv = [torch.zeros_like(U0[0]) for _ in range(nvar)], torch.zeros_like(U0[0])
    B = _BH(lay, bh, t + (dt if stage else 0.0)) if bh else None
    for d in range(3):
        pairs = [_x_faces(p, _x_pad(q, lay, d, 3), d) for q in W]
        L = [_x_sl(hi, d, 0, -1) for _, hi in pairs]
        R = [_x_sl(lo, d, 1, 0) for lo, _ in pairs]
        F, vf = _x_riemann(p, d, L, R)
        if B is not None:
            X = B.inside(d)
            xl, xr = _x_sl(X, d, 0, -1), _x_sl(X, d, 1, 0)
            cut = (xl != xr) & ~torch.where(xr, F[0] > 0, F[0] < 0)
            F = [torch.where(cut, torch.zeros_like(f), f) for f in F]
            if vf is not None:
                vf = torch.where(cut, torch.zeros_like(vf), vf)
        idx = 1.0 / lay.dx[d]
        for q in range(nvar):
            acc[q] = acc[q] - (_x_sl(F[q], d, 1, 0) - _x_sl(F[q], d, 0, -1)) * idx
        if p.dual:
            dv = dv + (_x_sl(vf, d, 1, 0) - _x_sl(vf, d, 0, -1)) * idx
        if B is not None:
            ph = B.phi(d)
            m, c, q = _x_sl(ph, d, 0, -2), _x_sl(ph, d, 1, -1), _x_sl(ph, d, 2, 0)
            acc[1 + d] = acc[1 + d] - W[0] * (q - m) * (0.5 * idx)
            acc[4] = acc[4] - (_x_sl(F[0], d, 1, 0) * (q - c) + _x_sl(F[0], d, 0, -1) * (c - m)) * (0.5 * idx)
    out = [u0 + dt * a if stage == 0 else 0.5 * (u0 + (ui + dt * a)) for u0, ui, a in zip(U0, Uin, acc)]
    out[0] = torch.clamp(out[0], min=p.rho_floor)
    if p.dual:
        h = dt if stage == 0 else 0.5 * dt
        if p.eos:
            P, _, _ = _x_closure(p, out[0], out[5])
            out[5] = out[5] - P * dv * h
        else:
            out[5] = out[5] * torch.exp(-(p.gamma - 1) * dv * h)
        out[5] = torch.clamp(out[5], min=p.u_floor)
    return torch.stack(out)


def _x_step(lay, W, par, bh):
    p = _Params(par)
    U0 = _x_p2c(p, W)
    P = _x_c2p(p, U0)
    cs = torch.sqrt((P[6] if p.eos else p.gamma) * P[4] / P[0])
    lim = torch.stack([lay.dx[a] / (P[1 + a].abs() + cs) for a in range(3)]).amin(0)
    if bh:
        B = _BH(lay, bh, 0.0)
        r2 = B.r2()
        gr = bh["GM"] * torch.sqrt(r2) / (r2 + bh["r_soft"] ** 2) ** 1.5
        lim = torch.minimum(lim, torch.sqrt(min(lay.dx) / gr))
        lim = torch.where(B.inside(), torch.full_like(lim, float("inf")), lim)
    dt = CFL * float(lim.min())
    U1 = _x_stage(p, lay, bh, 0, U0, U0, dt, 0.0)
    U = _x_stage(p, lay, bh, 1, U0, U1, dt, 0.0)
    if bh:
        X = _BH(lay, bh, dt).inside()
        fl = [p.rho_floor, 0.0, 0.0, 0.0, p.u_floor, p.u_floor]
        U = torch.stack([torch.where(X, torch.full_like(u, fl[q]), u) for q, u in enumerate(U)])
    if p.dual:
        E = U[4]
        for d in range(3):
            E = _x_pad(E, lay, d, 1)
        emax = torch.nn.functional.max_pool3d(E[None, None], 3, stride=1)[0, 0]
        r = torch.clamp(U[0], min=p.rho_floor)
        Uc = U[4] - 0.5 * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / r
        U[5] = torch.where((Uc > 0) & (Uc > p.eta2 * emax), Uc, U[5])
    S = _pack(lay, U)
    if p.dual:   # the resynchronisation leaves the energy's ghost cells filled
        S[4] = _x_filled(lay, U[4])
    return {"U": S, "dt": torch.tensor([dt], dtype=torch.float64)}


def _x_filled(lay, A):
    """A global field in the MeshBlock layout, ghost cells by the boundaries."""
    out = torch.zeros(lay.ntot, dtype=torch.float64, device=DEV)
    for b in range(lay.nb):
        idx = []
        for a in range(3):
            g = lay.gofs(a)
            i = torch.arange(int(lay.pd[b][a]), device=DEV) + int(lay.blocks[b][a]) - g
            idx.append(i % lay.N[a] if lay.bc[a] == 1 else torch.clamp(i, 0, lay.N[a] - 1))
        out[int(lay.off[b]):int(lay.off[b + 1])] = A[idx[2]][:, idx[1]][:, :, idx[0]].reshape(-1)
    return out


def _x_gravity(lay, rho):
    """The periodic seven-point Poisson problem by FFT (zero-mean potential)."""
    S = -4 * np.pi * G_CODE * rho
    S = S - S.mean()
    lam = 0.0
    for a, k in ((0, 2), (1, 1), (2, 0)):
        n = lay.N[a]
        th = 2 * np.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n
        lam = lam + ((2 - 2 * torch.cos(th)) / lay.dx[a] ** 2).reshape([-1 if q == k else 1 for q in range(3)])
    H = torch.fft.fftn(S)
    lam[0, 0, 0] = 1.0
    H = H / lam
    H[0, 0, 0] = 0.0
    return torch.fft.ifftn(H).real.contiguous()


def _x_axis(src, dst, a):
    """[N_dst, N_src] weights of the sample average along a, and the inside fraction."""
    n, m = dst.N[a], src.N[a]
    Wt = torch.zeros((n, m), dtype=torch.float64, device=DEV)
    f = torch.zeros(n, dtype=torch.float64, device=DEV)
    rows = torch.arange(n, device=DEV)
    for o in (-0.25, 0.25):
        x = dst.xmin[a] + (rows.double() + 0.5 + o) * dst.dx[a]
        ins = ((x >= src.xmin[a]) & (x <= src.xmin[a] + m * src.dx[a])).double()
        u = (x - src.xmin[a]) / src.dx[a] - 0.5
        i = torch.floor(u)
        t = u - i
        for k, w in ((i, 1 - t), (i + 1, t)):
            Wt.index_put_((rows, torch.clamp(k.long(), 0, m - 1)), 0.5 * ins * w, accumulate=True)
        f += 0.5 * ins
    return Wt, f


def _x_remap(src, dst, W):
    U = _x_p2c(_Params(dict(dual=1)), W)
    A = [_x_axis(src, dst, a) for a in range(3)]
    G = U[[0, 1, 2, 3, 5]]
    for a, k in ((0, 3), (1, 2), (2, 1)):
        G = torch.movedim(torch.movedim(G, k, -1) @ A[a][0].T, -1, k)
    fl = 1.0 - A[0][1][None, None, :] * A[1][1][None, :, None] * A[2][1][:, None, None]
    G[0] += fl * 1e-8
    G[4] += fl * 1e-10
    ke = 0.5 * (G[1] ** 2 + G[2] ** 2 + G[3] ** 2) / G[0]
    return {"U": _pack(dst, torch.stack([G[0], G[1], G[2], G[3], G[4] + ke, G[4]]))}


def exact(case, seed):
    """What run() returns, in plain torch.  None for a window of local steps (thousands
    of block updates: minutes here), for an isolated solve (a dense boundary problem)
    and for training (its weights are rounded to 16 bits after every step)."""
    f = case["family"]
    if f in STEPS:
        return _x_step(*STEPS[f](case, seed))
    if f == "eos":
        T, P, c2, _, _ = _x_invert(*_eos_inputs(case, seed))
        return {"T": T, "P": P, "cs2": c2}
    if f == "gravity" and not case["isolated"]:
        lay, W = _gravity_setup(case, seed)
        return {"phi": _x_gravity(lay, W[0]), "cycles": None}
    if f == "remap":
        return _x_remap(*_remap_setup(case, seed))
    return None
