"""Atoms on one straight line.  A torsion over four of them has no plane on either side: both of its
normals are zero, and the terms must stay finite (its forces vanish with the normals).

With zero torsion barriers such a torsion adds nothing, so energies and forces compare with the FP64 oracle's
for the chain without torsions, within the bounds of the force tests (1e-5 relative, 1e-4 kcal/mol)."""
import dataclasses

import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

from systems import gpu_context, oracle_system, raw_grids32, state_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _chain(n, barrier):
    """n atoms 1.25 A apart along x (differences and cross products are exact in FP32), with every bond,
    angle (at rest when straight) and torsion of the chain."""
    i = np.arange(n)
    col = lambda m, k: np.stack([i[:m] + d for d in range(k)], 1).astype(np.int32)
    bonds, angles, torsions = col(n - 1, 2), col(n - 2, 3), col(n - 3, 4)
    x0 = np.zeros((n, 3))
    x0[:, 0] = 1.25 * (i - (n - 1) / 2)
    return S.Ligand(mass=np.full(n, 12.011), charge=np.where(i % 2, 0.2, -0.2) * (n % 2 == 0), rstar=np.full(n, 1.8),
                    eps=np.full(n, 0.1), bonds=bonds, bond_k=np.full(n - 1, 400.0), bond_r0=np.full(n - 1, 1.3),
                    angles=angles, angle_k=np.full(n - 2, 60.0), angle_theta0=np.full(n - 2, np.pi), torsions=torsions,
                    torsion_V=np.full((n - 3, 3), barrier), torsion_gamma=np.tile([0.0, np.pi, 0.0], (n - 3, 1)), x0=x0)


def _setup(lig):
    sys_ = dataclasses.replace(S.config_small(1), ligand=lig)
    g32 = raw_grids32(sys_)
    T, alpha, dt = state_table(sys_)
    K = len(T)
    x = np.repeat(lig.x0[None], K, 0).astype(np.float32)
    x[..., 2] += np.linspace(0.0, 2.0, K, dtype=np.float32)[:, None]  # along z: the chain stays on its line
    return sys_, g32, T, alpha, dt, gpu_context(sys_, g32, T, alpha, dt), x, np.arange(K, dtype=np.int32)


@pytest.mark.parametrize("n", [4, 8])
@pytest.mark.parametrize("barrier", [0.0, 1.5])
def test_energies_and_forces_of_a_straight_chain(n, barrier):
    sys_, g32, T, alpha, dt, ctx, x, states = _setup(_chain(n, barrier))
    xd, sd = torch.from_numpy(x).cuda(), torch.from_numpy(states).cuda()
    F = torch.full_like(xd, float("nan"))
    comps = torch.full((len(x), 4), float("nan"), dtype=torch.float64, device="cuda")
    ctx.energy_force(sd, xd, F, comps)
    re = torch.full_like(comps, float("nan"))
    ctx.reduced_energies(len(x), x=xd, comps=re)
    F, comps, re = F.cpu().numpy(), comps.cpu().numpy(), re.cpu().numpy()
    assert np.isfinite(F).all() and np.isfinite(comps).all()
    assert np.all(np.abs(re - comps) <= 1e-5 * np.abs(comps) + 1e-4)
    if barrier:
        return
    none = dataclasses.replace(sys_.ligand, torsions=np.zeros((0, 4), np.int32), torsion_V=np.zeros((0, 3)),
                               torsion_gamma=np.zeros((0, 3)))
    osys = oracle_system(sys_, g32, T, alpha, dt, ligand=none)
    w_sg, w_g, _ = osys.state_weights()
    for k in range(len(x)):
        co, Fo = osys.energy_force(x[k].astype(np.float64), w_sg[k], w_g[k])
        assert np.all(np.abs(comps[k] - co) <= 1e-5 * np.abs(co) + 1e-4)
        assert np.linalg.norm(F[k] - Fo) <= 1e-5 * np.linalg.norm(Fo)


@pytest.mark.parametrize("n", [4, 8, 40])
def test_trials_of_a_straight_chain_can_be_accepted(n):
    """The starting energy of a trial is finite, so some of the replicas move (a trial that starts from a NaN
    is always rejected).  40 atoms: two warps per replica; in one ligand's launch and in a batch."""
    from paper_1507_03703_gb300.algdock import Context
    lig = _chain(n, 1.5)
    lig = dataclasses.replace(lig, charge=np.zeros(n))
    sys_, g32, T, alpha, dt, ctx, x, states = _setup(lig)
    batch = Context(0)
    batch.grids_load(sys_.grid, *g32, ligand=lig)
    batch.states_set(T, alpha, dt)
    batch.batch_load([lig], sys_.site)
    batch.batch_layout(np.zeros(len(x), dtype=np.int32), n)
    for c, trial in ((ctx, ctx.hmc_cycle), (batch, batch.batch_hmc_cycle)):
        xd, sd = torch.from_numpy(x).cuda(), torch.from_numpy(states).cuda()
        comps = torch.full((len(x), 4), float("nan"), dtype=torch.float64, device="cuda")
        dH = torch.full((len(x),), float("nan"), dtype=torch.float64, device="cuda")
        acc = torch.zeros(len(x), dtype=torch.uint8, device="cuda")
        trial(sd, xd, comps, dH, acc, n_steps=2, seed=5, cycle=1)
        assert torch.isfinite(comps).all() and torch.isfinite(dH).all()
        assert acc.any()
