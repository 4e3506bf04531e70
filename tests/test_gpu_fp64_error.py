"""The all-FP64 path's rounding error against extended precision: no more than a plain FP64 evaluation with
square roots and divisions makes (root mean square over configurations, with a tenth for the order of sums).

Bonds alone (a bond's stretch is a few hundredths of its length, so the length's rounding counts many times) and
pairs alone (r^-12 counts that of 1/r^2 six times), on lattices of zeros without a restraint in reach."""
import dataclasses

import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if np.finfo(np.longdouble).eps > 2.0 ** -62:
    pytest.skip("no extended precision on this host", allow_module_level=True)


def _separation(lig):
    D = np.full((lig.n_atoms,) * 2, 99)
    np.fill_diagonal(D, 0)
    D[lig.bonds[:, 0], lig.bonds[:, 1]] = D[lig.bonds[:, 1], lig.bonds[:, 0]] = 1
    for k in range(lig.n_atoms):
        D = np.minimum(D, D[:, k, None] + D[None, k])
    return D


def _evaluate(lig, x, T, bonds):
    """U_L and forces of the bonds or of the pairs, every operation in T."""
    x = x.astype(T)
    F, E = np.zeros_like(x), np.zeros(len(x), T)
    if bonds:
        for (i, j), k, r0 in zip(lig.bonds, lig.bond_k.astype(T), lig.bond_r0.astype(T)):
            d = x[:, i] - x[:, j]
            r = np.sqrt((d * d).sum(-1))
            E += k * (r - r0) ** 2
            f = (-2 * k * (r - r0) / r)[:, None] * d
            F[:, i] += f
            F[:, j] -= f
        return E, F
    D, rstar, eps, q = _separation(lig), lig.rstar.astype(T), np.sqrt(lig.eps.astype(T)), lig.charge.astype(T)
    for i, j in zip(*np.nonzero(np.triu(D, 1) >= 3)):
        s_lj, s_el = (T(0.5), 1 / T(1.2)) if D[i, j] == 3 else (T(1), T(1))
        d = x[:, i] - x[:, j]
        r2 = (d * d).sum(-1)
        s2 = (rstar[i] + rstar[j]) ** 2 / r2
        s6 = s2 * s2 * s2
        e, el = s_lj * eps[i] * eps[j], s_el * T(332.0637) * q[i] * q[j] / np.sqrt(r2)
        E += e * (s6 * s6 - 2 * s6) + el
        f = ((12 * e * (s6 * s6 - s6) + el) / r2)[:, None] * d
        F[:, i] += f
        F[:, j] -= f
    return E, F


@pytest.mark.parametrize("n_atoms", [12, 33, 48, 70])
@pytest.mark.parametrize("bonds", [True, False])
def test_rounding_error(n_atoms, bonds):
    from paper_1507_03703_gb300.algdock import Context
    lig = S.make_ligand(n_atoms, seed=2, min_sep=2.6 if n_atoms > 60 else None)
    lig = dataclasses.replace(lig, angle_k=0 * lig.angle_k, torsion_V=0 * lig.torsion_V)
    lig = dataclasses.replace(lig, eps=0 * lig.eps, charge=0 * lig.charge) if bonds else \
        dataclasses.replace(lig, bond_k=0 * lig.bond_k)
    rng = np.random.default_rng(n_atoms)
    x = (lig.x0[None] + 0.03 * rng.normal(size=(256, n_atoms, 3))).astype(np.float32)
    ctx = Context(0)
    zero = np.zeros((33, 33, 33))
    ctx.grids_load_f64(S.cube_grid(np.zeros(3), 0.5, 33), zero, zero, zero, vmax_e=5.0)
    ctx.ligand_load(lig, np.zeros(3))
    ctx.states_set(np.array([300.0]), np.array([np.nan]), np.array([2.0]))
    F = torch.empty(x.shape, dtype=torch.float64, device="cuda")
    comps = ctx.energy_force_f64(torch.from_numpy(x).cuda(), torch.zeros(len(x), dtype=torch.int32, device="cuda"),
                                 force=F)
    E0, F0 = _evaluate(lig, x, np.longdouble, bonds)
    E1, F1 = _evaluate(lig, x, np.float64, bonds)
    scale = np.sqrt((F0 ** 2).sum((1, 2)))
    force_error = lambda f: np.sqrt((((f - F0) ** 2).sum((1, 2)) / scale ** 2).mean())
    energy_error = lambda e: np.sqrt(((e - E0) ** 2).mean())
    assert force_error(F.cpu().numpy()) <= 1.1 * force_error(F1)
    assert energy_error(comps.cpu().numpy()[:, 0]) <= 1.1 * energy_error(E1)
