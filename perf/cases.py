"""Performance cases: what a user of the library has it do, over the range of sizes it serves.

Each case is one pass through the public binding (``paper_1507_03703_gb300.algdock``).  ``listed``
gives the fixed cases, ``draw`` more of the same ranges, ``prepare`` the inputs and the loaded
context, ``run`` one pass, ``work`` the bytes and operations a pass cannot do without, and
``exact`` the same outputs in 64-bit torch where they are computed numbers.

The kinds of work:
  hmc       one HMC trial of every replica of a ladder (algdock_hmc_cycle)
  cycle     one iteration of the paper's loop: trial, external moves, exchange, snapshot
            (algdock_cycle)
  batch     one HMC trial of many ligands of uneven size (algdock_batch_hmc_cycle)
  ukn       re-evaluation of stored samples at every state (algdock_reduced_energies)
  mbar      the free energies of a ladder from its u_kn (algdock_mbar)
  eval64    energies and forces of the all-FP64 path (algdock_energy_force_f64)
  grids     the receptor's grids by direct sum (algdock_grids_build)
  train     one training step of the learned proposal (algdock_mlp_grad, algdock_mlp_adam)
  propose   learned proposals with their Metropolis test (algdock_propose_learned)
  endpoint  the end-point correction: target interaction and FEP (algdock_target_interaction,
            algdock_fep)
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1507_03703_gb300 import synthetic as S
from paper_1507_03703_gb300.algdock import (D0, K_RESTRAINT, MLP_DMAX, MLP_NFEAT, MLP_NPARAMS, VMAX_R, Context,
                                            pack_mlp)

KB = 0.0019872043        # kcal / (mol K)
COULOMB = 332.0637       # kcal A / (mol e^2)
VMAX_E = 5.0             # soft electrostatic cap, kcal / (mol e)
SITE = np.zeros(3)


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: a 20-atom ligand on the 33^3 grid, one replica per state of the 8 + 8
        # state test ladder, 20 steps; latency and launches count
        {"name": "hmc_small", "kind": "hmc", "atoms": 20, "grid": 33, "spacing": 0.5, "bc": 8, "cd": 8, "chains": 1,
         "steps": 20},
        # a large ligand with an odd atom count (three atoms per lane), a run of ordinary size
        {"name": "hmc_large_ligand", "kind": "hmc", "atoms": 83, "grid": 129, "spacing": 0.25, "bc": 16, "cd": 32,
         "chains": 24, "steps": 50},
        # the paper's loop at paper scale: 48 atoms, 32 + 96 states, 64 chains, 50 steps, 20 external
        # moves where the paper makes them, 25 exchange sweeps and the snapshot for MBAR
        {"name": "cycle_paper_scale", "kind": "cycle", "atoms": 48, "bc": 32, "cd": 96, "chains": 64, "steps": 50,
         "external": 20},
        # a virtual screen: 96 ligands of 10-70 atoms, 64 states each, one launch per size class
        {"name": "batch_screen", "kind": "batch", "ligands": 96, "bc": 16, "cd": 48, "steps": 50},
        # a finished run's samples evaluated again at all 128 states for MBAR
        {"name": "ukn_reevaluation", "kind": "ukn", "atoms": 48, "bc": 32, "cd": 96, "samples": 102400},
        # MBAR in full precision at the paper's size
        {"name": "mbar_fp64", "kind": "mbar", "states": 128, "per_state": 800, "mode": 0},
        # MBAR with compensated FP32 sums at the precision study's size
        {"name": "mbar_fp32", "kind": "mbar", "states": 256, "per_state": 3907, "mode": 2},
        # the precision study's FP64 arm over one snapshot of replicas
        {"name": "eval_fp64", "kind": "eval64", "atoms": 48, "bc": 32, "cd": 96, "samples": 8192},
        # a receptor's grids, once per receptor
        {"name": "grids_paper_scale", "kind": "grids", "grid": 129, "spacing": 0.25, "receptor": 4000},
        # one Adam step of the proposal network, forward and backward
        {"name": "learned_train", "kind": "train", "batch": 4096, "dims": 22},
        # a learned move of every chain, four times over, after an HMC cycle
        {"name": "learned_propose", "kind": "propose", "atoms": 48, "bc": 32, "cd": 96, "replicas": 4096, "moves": 4},
        # f_DE of a run's milestone samples against all receptor atoms
        {"name": "endpoint_fep", "kind": "endpoint", "atoms": 48, "receptor": 4000, "samples": 16384},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["hmc", "hmc", "cycle", "batch", "ukn", "mbar", "mbar", "eval64", "grids", "train", "propose",
                       "endpoint"])
    if kind == "hmc":
        small = rng.random() < 0.5
        return {"kind": kind, "atoms": rng.randint(5, 30 if small else 90), "grid": 33 if small else 129,
                "spacing": 0.5 if small else 0.25, "bc": rng.randint(4, 32), "cd": rng.randint(4, 64),
                "chains": _log_int(rng, 1, 24), "steps": rng.choice([10, 20, 50])}
    if kind == "cycle":
        return {"kind": kind, "atoms": rng.randint(20, 60), "bc": rng.randint(4, 32), "cd": rng.randint(8, 96),
                "chains": _log_int(rng, 4, 64), "steps": rng.choice([20, 50]), "external": rng.choice([0, 20])}
    if kind == "batch":
        return {"kind": kind, "ligands": _log_int(rng, 8, 96), "bc": rng.randint(4, 16), "cd": rng.randint(8, 48),
                "steps": rng.choice([20, 50])}
    if kind == "ukn":
        return {"kind": kind, "atoms": rng.randint(10, 80), "bc": rng.randint(4, 32), "cd": rng.randint(8, 96),
                "samples": _log_int(rng, 1000, 60000)}
    if kind == "mbar":
        return {"kind": kind, "states": rng.randint(16, 256), "per_state": _log_int(rng, 50, 1500),
                "mode": rng.choice([0, 0, 1, 2])}
    if kind == "eval64":
        return {"kind": kind, "atoms": rng.randint(10, 72), "bc": rng.randint(4, 32), "cd": rng.randint(8, 96),
                "samples": _log_int(rng, 100, 8192)}
    if kind == "grids":
        return {"kind": kind, "grid": rng.randint(25, 110), "spacing": rng.choice([0.25, 0.375, 0.5]),
                "receptor": _log_int(rng, 300, 4000)}
    if kind == "train":
        return {"kind": kind, "batch": _log_int(rng, 256, 16384), "dims": rng.randint(6, 22)}
    if kind == "propose":
        return {"kind": kind, "atoms": rng.randint(12, 60), "bc": rng.randint(4, 32), "cd": rng.randint(8, 96),
                "replicas": _log_int(rng, 100, 8192), "moves": rng.randint(1, 4)}
    return {"kind": kind, "atoms": rng.randint(10, 70), "receptor": _log_int(rng, 300, 4000),
            "samples": _log_int(rng, 500, 10000)}


# ------------------------------------------------------------------ systems (kept per process)
@functools.lru_cache(maxsize=None)
def _ligand(atoms):
    return S.make_ligand(atoms, seed=2, min_sep=2.6 if atoms > 60 else None)


@functools.lru_cache(maxsize=None)
def _receptor(n, pocket=7.0):
    return S.make_receptor(n, SITE, 2, pocket_radius=pocket)


@functools.lru_cache(maxsize=2)
def _batch_system(n_ligands):
    sys_, ligs = S.config_batch(3, n_ligands=n_ligands)
    return sys_.receptor, ligs


@functools.lru_cache(maxsize=4)
def _raw_grids(n_rec, pocket, grid_n, spacing):
    """A receptor's raw grids by direct sum in torch, float64 sums of float32 terms, [n]^3."""
    rec, grid = _receptor(n_rec, pocket), S.cube_grid(SITE, spacing, grid_n)
    out = _direct_sum(rec, grid, torch.float32, 2048)
    return tuple(a.float() for a in out)


def _direct_sum(rec, grid, dtype, chunk):
    dev = "cuda"
    ax = [torch.as_tensor(grid.origin[d] + grid.spacing * np.arange(grid.n[d]), device=dev) for d in range(3)]
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    nodes = torch.stack([x, y, z], -1).reshape(-1, 3)
    pos = torch.as_tensor(rec.xyz, device=dev)
    two_r = 2.0 * torch.as_tensor(rec.rstar, device=dev)
    eps = torch.as_tensor(rec.eps, device=dev)
    sA, sB = (eps.sqrt() * two_r ** 6).to(dtype), ((2.0 * eps).sqrt() * two_r ** 3).to(dtype)
    q4 = (0.25 * torch.as_tensor(rec.charge, device=dev)).to(dtype)
    ljr, lja, elec = (torch.empty(nodes.shape[0], dtype=torch.float64, device=dev) for _ in range(3))
    for b in range(0, nodes.shape[0], chunk):
        r2 = _r2(nodes[b:b + chunk], pos, dtype)
        i2 = 1.0 / r2.clamp(min=1e-4)
        ljr[b:b + chunk] = torch.sum((i2 * i2 * i2).square_().mul_(sA), -1, dtype=torch.float64)
        i2 = 1.0 / r2.clamp(min=4.0)
        lja[b:b + chunk] = -torch.sum((i2 * i2 * i2).mul_(sB), -1, dtype=torch.float64)
        elec[b:b + chunk] = COULOMB * torch.sum(i2.mul_(q4), -1, dtype=torch.float64)
    shape = (grid.n[2], grid.n[1], grid.n[0])
    return ljr.reshape(shape), lja.reshape(shape), elec.reshape(shape)


def _r2(p, pos, dtype):
    r2 = (p[:, None, 0] - pos[None, :, 0]).to(dtype).square_()
    r2 += (p[:, None, 1] - pos[None, :, 1]).to(dtype).square_()
    r2 += (p[:, None, 2] - pos[None, :, 2]).to(dtype).square_()
    return r2


def _ladder(bc, cd):
    legs = [S.bc_ladder(bc), S.cd_ladder(cd)]
    return tuple(np.concatenate([getattr(leg, f) for leg in legs]) for f in ("T", "alpha", "dt_fs"))


def _poses(lig, rec, n, seed, tries=6, jitter=0.03):
    """n placements in the pocket (of `tries` random ones the farthest from the receptor), with
    thermal distortions of `jitter` A, as float32 [n][atoms][3] on the device."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    pos = torch.as_tensor(rec.xyz, device="cuda", dtype=torch.float32)
    pos = pos[pos.norm(dim=1).argsort()[:400]]
    x0 = torch.as_tensor(lig.x0, device="cuda", dtype=torch.float32)
    best = torch.empty((n, lig.n_atoms, 3), device="cuda")
    best_d = torch.full((n,), -1.0, device="cuda")
    for _ in range(tries):
        q = torch.randn((n, 4), device="cuda", generator=g)
        w, a, b, c = (q / q.norm(dim=1, keepdim=True)).unbind(1)
        R = torch.stack([1 - 2 * (b * b + c * c), 2 * (a * b - w * c), 2 * (a * c + w * b),
                         2 * (a * b + w * c), 1 - 2 * (a * a + c * c), 2 * (b * c - w * a),
                         2 * (a * c - w * b), 2 * (b * c + w * a), 1 - 2 * (a * a + b * b)], 1).reshape(n, 3, 3)
        off = torch.randn((n, 3), device="cuda", generator=g)
        off = off / off.norm(dim=1, keepdim=True)
        off = off * (5.5 * torch.rand((n, 1), device="cuda", generator=g) ** (1.0 / 3.0))
        off[:, 2].abs_()
        x = torch.einsum("ai,nji->naj", x0, R) + off[:, None, :]
        for s in range(0, n, 4096):
            xc = x[s:s + 4096]
            d = torch.full((xc.shape[0],), 99.0, device="cuda")
            for i in range(lig.n_atoms):
                d = torch.minimum(d, (xc[:, i, None, :] - pos[None]).square().sum(-1).min(dim=1).values)
            better = d > best_d[s:s + 4096]
            best[s:s + 4096][better] = xc[better]
            best_d[s:s + 4096][better] = d[better]
    return (best + jitter * torch.randn(best.shape, device="cuda", generator=g)).contiguous()


def _context(case, lig, rec_n=4000):
    ctx = Context(0)
    n, h = case.get("grid", 129), case.get("spacing", 0.25)
    rec_n = 1500 if n == 33 else rec_n
    ctx.grids_load(S.cube_grid(SITE, h, n), *_raw_grids(rec_n, 7.0, n, h), vmax_e=VMAX_E)
    ctx.ligand_load(lig, SITE)
    T, alpha, dt = _ladder(case["bc"], case["cd"])
    ctx.states_set(T, alpha, dt)
    return ctx, _receptor(rec_n)


def _states(case, n):
    return (torch.arange(n, device="cuda") % (case["bc"] + case["cd"])).to(torch.int32)


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    s = {"case": case, "kind": case["kind"], "seed": seed & 0x7FFFFFFF, "cycle": 0}
    return globals()["_prepare_" + case["kind"]](case, seed, s)


def _hmc_arrays(s, n):
    s["comps"] = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    s["dH"] = torch.zeros(n, dtype=torch.float64, device="cuda")
    s["accepted"] = torch.zeros(n, dtype=torch.uint8, device="cuda")
    s["counters"] = torch.zeros(4, dtype=torch.int64, device="cuda")


def _prepare_hmc(case, seed, s):
    lig = _ligand(case["atoms"])
    s["ctx"], rec = _context(case, lig)
    n = case["chains"] * (case["bc"] + case["cd"])
    s["x"] = _poses(lig, rec, n, seed)
    s["state_of"] = torch.cat([torch.arange(b, b + k, device="cuda").repeat(case["chains"])
                               for b, k in ((0, case["bc"]), (case["bc"], case["cd"]))]).to(torch.int32)
    _hmc_arrays(s, n)
    return s


def _prepare_cycle(case, seed, s):
    _prepare_hmc(case, seed, s)
    c, K = case["chains"], (case["bc"], case["cd"])
    s["legs"] = [(K[0], 0), (K[1], K[0])]
    s["config_of"] = torch.cat([torch.arange(k, device="cuda").repeat(c) for k in K]).to(torch.int32)
    s["u_kn"] = torch.zeros(c * (K[0] ** 2 + K[1] ** 2), dtype=torch.float64, device="cuda")
    return s


def _prepare_batch(case, seed, s):
    rec, ligs = _batch_system(case["ligands"])
    grid = S.cube_grid(SITE, 0.25, 129)
    s["ctx"] = ctx = Context(0)
    ctx.grids_load(grid, *_raw_grids(4000, 11.0, 129, 0.25), vmax_e=VMAX_E)
    ctx.states_set(*_ladder(case["bc"], case["cd"]))
    ctx.batch_load(ligs, SITE)
    K, stride = case["bc"] + case["cd"], max(lig.n_atoms for lig in ligs)
    ctx.batch_layout(np.repeat(np.arange(len(ligs)), K), stride)
    n = len(ligs) * K
    s["x"] = torch.zeros((n, stride, 3), dtype=torch.float32, device="cuda")
    for i, lig in enumerate(ligs):
        s["x"][i * K:(i + 1) * K, :lig.n_atoms] = _poses(lig, rec, K, seed + 7919 * i, tries=3)
    s["state_of"] = torch.arange(K, device="cuda").repeat(len(ligs)).to(torch.int32)
    _hmc_arrays(s, n)
    return s


def _prepare_ukn(case, seed, s):
    lig = _ligand(case["atoms"])
    s["ctx"], rec = _context(case, lig)
    base = _poses(lig, rec, 4096, seed)
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    n, K = case["samples"], case["bc"] + case["cd"]
    pick = torch.randint(0, base.shape[0], (n,), device="cuda", generator=g)
    x = base[pick]
    s["x"] = (x + 0.02 * torch.randn(x.shape, device="cuda", generator=g)).contiguous()
    s["comps"] = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    s["u_kn"] = torch.zeros((K, n), dtype=torch.float64, device="cuda")
    return s


def _prepare_mbar(case, seed, s):
    """Samples of a temperature ladder: energies from gamma distributions of 60 degrees of freedom,
    reduced by inverse temperatures a factor of two apart at the ends (300 and 600 K)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    K, n = case["states"], case["per_state"]
    beta = 0.5 ** (torch.arange(K, device="cuda", dtype=torch.float64) / (K - 1))
    E = -torch.log(torch.rand((30, K, n), device="cuda", dtype=torch.float64, generator=g)).sum(0) / beta[:, None]
    E = E.reshape(-1)
    s["ctx"] = Context(0)
    s["u_kn"] = torch.outer(beta, E)
    s["N_k"] = np.full(K, n, dtype=np.int64)
    return s


def _prepare_eval64(case, seed, s):
    lig = _ligand(case["atoms"])
    s["ctx"], rec = _context(case, lig)
    s["ctx"].grids_load_f64(S.cube_grid(SITE, 0.25, 129), *(a.double() for a in _raw_grids(4000, 7.0, 129, 0.25)),
                            vmax_e=VMAX_E)
    n = case["samples"]
    s["x"] = _poses(lig, rec, n, seed)
    s["state_of"] = _states(case, n)
    s["force"] = torch.zeros((n, lig.n_atoms, 3), dtype=torch.float64, device="cuda")
    s["comps"] = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    return s


def _prepare_grids(case, seed, s):
    s["ctx"] = Context(0)
    s["receptor"] = S.make_receptor(case["receptor"], SITE, seed)
    s["grid"] = S.cube_grid(SITE, case["spacing"], case["grid"])
    s["out"] = [torch.zeros((case["grid"],) * 3, dtype=torch.float32, device="cuda") for _ in range(3)]
    return s


def _network(seed):
    flat, w = pack_mlp(S.mlp_init(seed & 0xFFFF))
    return torch.from_numpy(flat).cuda(), torch.from_numpy(w.view(np.int16)).cuda()


def _prepare_train(case, seed, s):
    s["ctx"] = Context(0)
    s["params"], s["wbf16"] = _network(seed)
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = case["batch"]
    s["feat"] = torch.randn((n, MLP_NFEAT), device="cuda", generator=g)
    s["delta"] = 0.5 * torch.randn((n, MLP_DMAX), device="cuda", generator=g)
    s["m"], s["v"], s["grad"] = (torch.zeros(MLP_NPARAMS, device="cuda") for _ in range(3))
    s["loss"] = torch.zeros(1, device="cuda")
    return s


def _prepare_propose(case, seed, s):
    lig = _ligand(case["atoms"])
    s["ctx"], rec = _context(case, lig)
    s["params"], s["wbf16"] = _network(seed)
    n = case["replicas"]
    s["x"] = _poses(lig, rec, n, seed)
    s["state_of"] = (case["bc"] + torch.arange(n, device="cuda") % case["cd"]).to(torch.int32)
    s["comps"] = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    s["ctx"].reduced_energies(n, x=s["x"], comps=s["comps"])
    s["accepted"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    return s


def _prepare_endpoint(case, seed, s):
    lig, rec = _ligand(case["atoms"]), _receptor(case["receptor"])
    s["ctx"] = Context(0)
    s["ctx"].ligand_load(lig, SITE)
    s["ctx"].receptor_load(rec)
    n = case["samples"]
    base = _poses(lig, rec, min(n, 2048), seed)
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    x = base[torch.arange(n, device="cuda") % base.shape[0]]
    s["x"] = (x + 0.02 * torch.randn(x.shape, device="cuda", generator=g)).contiguous()
    psi = _target64(lig, rec, s["x"], torch.float32)
    s["u_sampling"] = psi + 0.2 * torch.randn(n, device="cuda", dtype=torch.float64, generator=g)
    s["psi"] = torch.zeros(n, dtype=torch.float64, device="cuda")
    return s


# ------------------------------------------------------------------ run
def run(s):
    ctx, c, k = s["ctx"], s["case"], s["kind"]
    s["cycle"] += 1
    if k == "hmc":
        ctx.hmc_cycle(s["state_of"], s["x"], s["comps"], s["dH"], s["accepted"], n_steps=c["steps"], seed=s["seed"],
                      cycle=s["cycle"], counters=s["counters"])
        return {f: s[f] for f in ("x", "comps", "dH", "accepted", "counters")}
    if k == "cycle":
        ctx.cycle(s["legs"], c["chains"], s["cycle"], s["x"], s["comps"], s["state_of"], s["config_of"],
                  n_steps=c["steps"], seed=s["seed"], counters=s["counters"], u_kn=s["u_kn"], n_external=c["external"])
        return {f: s[f] for f in ("x", "comps", "state_of", "config_of", "counters", "u_kn")}
    if k == "batch":
        ctx.batch_hmc_cycle(s["state_of"], s["x"], s["comps"], s["dH"], s["accepted"], n_steps=c["steps"],
                            seed=s["seed"], cycle=s["cycle"], counters=s["counters"])
        return {f: s[f] for f in ("x", "comps", "dH", "accepted", "counters")}
    if k == "ukn":
        ctx.reduced_energies(c["samples"], x=s["x"], comps=s["comps"], k_begin=0, k_count=c["bc"] + c["cd"],
                             u_kn=s["u_kn"])
        return {"comps": s["comps"], "u_kn": s["u_kn"]}
    if k == "mbar":
        f, iters = ctx.mbar(s["u_kn"], s["N_k"], precision_mode=c["mode"], raise_on_nonconvergence=False)
        return {"f": f, "iterations": iters}
    if k == "eval64":
        ctx.energy_force_f64(s["x"], s["state_of"], s["force"], s["comps"])
        return {"force": s["force"], "comps": s["comps"]}
    if k == "grids":
        ctx.grids_build(s["grid"], s["receptor"], *s["out"])
        return {"ljr": s["out"][0], "lja": s["out"][1], "elec": s["out"][2]}
    if k == "train":
        ctx.mlp_grad(s["params"], s["wbf16"], s["feat"], s["delta"], c["dims"], s["grad"], s["loss"])
        ctx.mlp_adam(s["params"], s["wbf16"], s["grad"], s["m"], s["v"], s["cycle"], 1e-3)
        return {f: s[f] for f in ("grad", "loss", "params", "wbf16", "m", "v")}
    if k == "propose":
        ctx.propose_learned(s["params"], s["wbf16"], s["state_of"], s["x"], s["comps"], c["moves"], seed=s["seed"],
                            cycle=s["cycle"], accepted=s["accepted"])
        return {f: s[f] for f in ("x", "comps", "accepted")}
    ctx.target_interaction(s["x"], s["psi"])
    r = ctx.fep(s["psi"], s["u_sampling"], beta=1.0 / (KB * 300.0))
    return {"psi": s["psi"], "f": r["f"], "sigma": r["sigma"], "n_eff": r["n_eff"]}


# ------------------------------------------------------------------ work
def _bond_distance(lig):
    n = lig.n_atoms
    d = np.full((n, n), 99)
    np.fill_diagonal(d, 0)
    adj = np.zeros((n, n), dtype=bool)
    for a, b in lig.bonds:
        adj[a, b] = adj[b, a] = True
    reach = np.eye(n, dtype=bool)
    for step in (1, 2, 3):
        new = (reach @ adj) & (d == 99)
        d[new] = step
        reach = new
    return d


@functools.lru_cache(maxsize=None)
def _eval_flops(atoms):
    """One force evaluation: 26 per nonbonded pair, 20 / 60 / 100 per bond / angle / torsion, 170
    per atom for the five interpolated channels and 12 for the integrator."""
    return _lig_flops(_ligand(atoms))


def _lig_flops(lig):
    pairs = int((np.triu(_bond_distance(lig), 1) > 2).sum())
    return 26 * pairs + 20 * len(lig.bonds) + 60 * len(lig.angles) + 100 * len(lig.torsions) + 182 * lig.n_atoms


def work(case):
    k = case["kind"]
    K = case.get("bc", 0) + case.get("cd", 0)
    if k in ("hmc", "cycle"):
        n = case["chains"] * K
        byts = n * (24 * case["atoms"] + 77)
        fl = n * (case["steps"] + 1) * _eval_flops(case["atoms"])
        if k == "cycle":
            byts += 8 * case["chains"] * (case["bc"] ** 2 + case["cd"] ** 2) + 16 * n
        return {"bytes": byts, "flops": fl}
    if k == "batch":
        ligs = _batch_system(case["ligands"])[1]
        return {"bytes": sum(K * (24 * lig.n_atoms + 77) for lig in ligs),
                "flops": sum(K * (case["steps"] + 1) * _lig_flops(lig) for lig in ligs)}
    if k == "ukn":
        return {"bytes": case["samples"] * (12 * case["atoms"] + 32 + 8 * K),
                "flops": case["samples"] * (_eval_flops(case["atoms"]) + 5 * K)}
    if k == "mbar":  # the samples read once; some 40 iterations of two passes, an operation pair per element
        n = case["states"] * case["per_state"]
        return {"bytes": 8 * case["states"] * (n + 2), "flops": 40 * 4 * case["states"] * n}
    if k == "eval64":
        return {"bytes": case["samples"] * (36 * case["atoms"] + 36),
                "flops": case["samples"] * _eval_flops(case["atoms"])}
    if k == "grids":
        return {"bytes": 12 * case["grid"] ** 3 + 48 * case["receptor"],
                "flops": 20 * case["grid"] ** 3 * case["receptor"]}
    if k == "train":
        return {"bytes": case["batch"] * 4 * (MLP_NFEAT + case["dims"]) + 22 * MLP_NPARAMS,
                "flops": 3 * case["batch"] * 2 * MLP_NPARAMS}
    if k == "propose":
        n = case["replicas"]
        return {"bytes": n * (24 * case["atoms"] + 72) + 6 * MLP_NPARAMS,
                "flops": n * case["moves"] * (2 * 2 * MLP_NPARAMS + _eval_flops(case["atoms"]))}
    return {"bytes": case["samples"] * (12 * case["atoms"] + 16) + 48 * case["receptor"],
            "flops": 18 * case["samples"] * case["atoms"] * case["receptor"]}


# ------------------------------------------------------------------ exact values in 64 bits
def _target64(lig, rec, x, dtype):
    """Receptor-ligand energy of configurations x by direct sum, terms in dtype, sums in 64 bits."""
    pos = torch.as_tensor(rec.xyz, device="cuda")
    two_r, eps = 2.0 * torch.as_tensor(rec.rstar, device="cuda"), torch.as_tensor(rec.eps, device="cuda")
    A, B = (eps.sqrt() * two_r ** 6).to(dtype), ((2 * eps).sqrt() * two_r ** 3).to(dtype)
    Q = torch.as_tensor(0.25 * rec.charge, device="cuda").to(dtype)
    psi = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
    for i in range(lig.n_atoms):
        r1 = 2.0 * lig.rstar[i]
        a, b = math.sqrt(lig.eps[i]) * r1 ** 6, math.sqrt(2 * lig.eps[i]) * r1 ** 3
        for s in range(0, x.shape[0], 4096):
            r2 = _r2(x[s:s + 4096, i].double(), pos, dtype)
            i2 = 1.0 / r2.clamp(min=1e-4)
            e = a * torch.sum((i2 * i2 * i2).square_().mul_(A), -1, dtype=torch.float64)
            i2 = i2.clamp_(max=0.25)
            e -= b * torch.sum((i2 * i2 * i2).mul_(B), -1, dtype=torch.float64)
            e += COULOMB * lig.charge[i] * torch.sum(i2.mul_(Q), -1, dtype=torch.float64)
            psi[s:s + 4096] += e
    return psi


def _interpolate(lat, grid, x):
    """Trilinear value of lattice [nz][ny][nx] at x [..., 3], clamped to the lattice."""
    o = torch.as_tensor(grid.origin, device="cuda")
    top = torch.as_tensor([n - 1.0 for n in grid.n], device="cuda")
    u = torch.minimum(torch.clamp((x - o) / grid.spacing, min=0.0), top)
    c = torch.minimum(u.detach().floor(), top - 1).long()
    t = u - c
    v = 0.0
    for k in range(8):
        b = [(k >> d) & 1 for d in range(3)]
        w = 1.0
        for d in range(3):
            w = w * (t[..., d] if b[d] else 1.0 - t[..., d])
        v = v + w * lat[c[..., 2] + b[2], c[..., 1] + b[1], c[..., 0] + b[0]]
    return v


def _components64(lig, raw, grid, x):
    """[N][4] energies (ligand, restraint, soft grid, hard grid) in 64 bits, differentiable in x."""
    dev = "cuda"
    t = lambda a: torch.as_tensor(np.asarray(a), device=dev)  # noqa: E731
    e = 0.0
    if len(lig.bonds):
        i, j = t(lig.bonds.astype(np.int64)).T
        r = (x[:, i] - x[:, j]).norm(dim=-1)
        e = e + (t(lig.bond_k) * (r - t(lig.bond_r0)) ** 2).sum(-1)
    if len(lig.angles):
        i, j, k = t(lig.angles.astype(np.int64)).T
        u, w = x[:, i] - x[:, j], x[:, k] - x[:, j]
        cs = ((u * w).sum(-1) / torch.sqrt((u * u).sum(-1) * (w * w).sum(-1))).clamp(-1.0, 1.0)
        e = e + (t(lig.angle_k) * (torch.acos(cs) - t(lig.angle_theta0)) ** 2).sum(-1)
    if len(lig.torsions):
        i, j, k, m = t(lig.torsions.astype(np.int64)).T
        b1, b2, b3 = x[:, j] - x[:, i], x[:, k] - x[:, j], x[:, m] - x[:, k]
        n1, n2 = torch.cross(b1, b2, dim=-1), torch.cross(b2, b3, dim=-1)
        phi = torch.atan2(b2.norm(dim=-1) * (b1 * n2).sum(-1), (n1 * n2).sum(-1))
        for h in range(3):
            e = e + (0.5 * t(lig.torsion_V)[:, h] * (1 + torch.cos((h + 1) * phi - t(lig.torsion_gamma)[:, h]))).sum(-1)
    dist = _bond_distance(lig)
    i, j = np.nonzero(np.triu(dist, 1) > 2)
    if len(i):
        far = t(dist[i, j] > 3)
        i, j = t(i), t(j)
        r2 = (x[:, i] - x[:, j]).square().sum(-1)
        s6 = ((t(lig.rstar)[i] + t(lig.rstar)[j]) ** 2 / r2) ** 3
        lj = torch.sqrt(t(lig.eps)[i] * t(lig.eps)[j]) * (s6 * s6 - 2 * s6)
        el = COULOMB * t(lig.charge)[i] * t(lig.charge)[j] / torch.sqrt(r2)
        e = e + (torch.where(far, 1.0, 0.5) * lj + torch.where(far, 1.0, 1.0 / 1.2) * el).sum(-1)
    mass = t(lig.mass)
    d = ((mass[:, None] * x).sum(1) / mass.sum()).norm(dim=-1)  # the site is the origin
    rest = 0.5 * K_RESTRAINT * torch.clamp(d - D0, min=0.0) ** 2
    v = raw[0].double().clamp(0.0, 1e10)
    hard = [v ** 0.25, raw[1].double(), raw[2].double()]
    soft = [(VMAX_R * torch.tanh(v / VMAX_R)) ** 0.25, VMAX_E * torch.tanh(raw[2].double() / VMAX_E)]
    two_r, eps, q = 2.0 * t(lig.rstar), t(lig.eps), t(lig.charge)
    sA, sB = eps.sqrt() * two_r ** 6, (2 * eps).sqrt() * two_r ** 3
    g = (sA * _interpolate(hard[0], grid, x) ** 4 + sB * _interpolate(hard[1], grid, x)
         + q * _interpolate(hard[2], grid, x)).sum(-1)
    sg = (sA * _interpolate(soft[0], grid, x) ** 4 + q * _interpolate(soft[1], grid, x)).sum(-1)
    if not torch.is_tensor(e):
        e = torch.zeros_like(g)
    return torch.stack([e, rest, sg, g], 1)


def _weights64(alpha):
    a = torch.as_tensor(alpha, device="cuda")
    s2 = (2 * a - 1) ** 2
    w = torch.stack([1 - s2, s2 * torch.sigmoid(1000.0 * (a - 0.5))])
    return torch.where(torch.isnan(a), torch.zeros_like(w), w)


def exact(case, seed):
    k = case["kind"]
    if k in ("ukn", "eval64"):
        s = prepare(case, seed)
        lig, grid, raw = _ligand(case["atoms"]), S.cube_grid(SITE, 0.25, 129), _raw_grids(4000, 7.0, 129, 0.25)
        T, alpha, _ = _ladder(case["bc"], case["cd"])
        w_sg, w_g = _weights64(alpha)
        comps, force = [], []
        for b in range(0, case["samples"], 2048):
            x = s["x"][b:b + 2048].double().requires_grad_(k == "eval64")
            c = _components64(lig, raw, grid, x)
            if k == "eval64":
                st = s["state_of"][b:b + 2048].long()
                u = c[:, 0] + c[:, 1] + w_sg[st] * c[:, 2] + w_g[st] * c[:, 3]
                force.append(-torch.autograd.grad(u.sum(), x)[0])
            comps.append(c.detach())
        comps = torch.cat(comps)
        if k == "eval64":
            return {"force": torch.cat(force), "comps": comps}
        beta = torch.as_tensor(1.0 / (KB * T), device="cuda")
        u = beta[:, None] * (comps[:, 0] + comps[:, 1] + w_sg[:, None] * comps[:, 2] + w_g[:, None] * comps[:, 3])
        return {"comps": comps, "u_kn": u}
    if k == "mbar":
        s = prepare(case, seed)
        W, n = s["u_kn"], torch.as_tensor(s["N_k"], device="cuda", dtype=torch.float64)
        W = W - W.min(0).values
        W.neg_().exp_()
        f = torch.zeros(W.shape[0], dtype=torch.float64, device="cuda")
        for _ in range(5000):
            new = -torch.log(W @ (1.0 / ((n * torch.exp(f)) @ W)))
            new -= new[0].clone()
            delta, f = float((new - f).abs().max()), new
            if delta < 1e-12:
                break
        return {"f": f.cpu().numpy(), "iterations": None}
    if k == "grids":
        s = prepare(case, seed)
        out = _direct_sum(s["receptor"], s["grid"], torch.float64, 4096)
        return {"ljr": out[0], "lja": out[1], "elec": out[2]}
    if k == "endpoint":
        s = prepare(case, seed)
        psi = _target64(_ligand(case["atoms"]), _receptor(case["receptor"]), s["x"], torch.float64)
        du = (psi - s["u_sampling"]) / (KB * 300.0)
        n, w = du.numel(), torch.exp(du.min() - du)
        n_eff = float(w.sum() ** 2 / (w * w).sum())
        return {"psi": psi, "f": float(du.min() - torch.log(w.mean())),
                "sigma": math.sqrt(max(n / n_eff - 1.0, 0.0) / (n - 1.0)), "n_eff": n_eff}
    return None
