"""The FP64 path at positions that are not finite: an atom at infinity has infinite bonds and no pairs (its
distant pairs add nothing), and a coordinate that is not a number reaches only what depends on it."""
import dataclasses

import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _evaluate(lig, x):
    from paper_1507_03703_gb300.algdock import Context
    ctx = Context(0)
    zero = np.zeros((9, 9, 9))
    ctx.grids_load_f64(S.cube_grid(np.zeros(3), 1.0, 9), zero, zero, zero, vmax_e=5.0)
    ctx.ligand_load(lig, np.zeros(3))
    ctx.states_set(np.array([300.0]), np.array([np.nan]), np.array([2.0]))
    xd = torch.from_numpy(x.astype(np.float32)).cuda()
    F = torch.zeros(x.shape, dtype=torch.float64, device="cuda")
    c = ctx.energy_force_f64(xd, torch.zeros(len(x), dtype=torch.int32, device="cuda"), force=F)
    return c.cpu().numpy(), F.cpu().numpy(), ctx.energy_force_f64(xd).cpu().numpy()


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_infinite_bond(sign):
    lig = S.make_ligand(2, seed=2)
    x = lig.x0[None].copy()
    x[0, 1, 2] = sign * np.inf
    for c in _evaluate(lig, x)[::2]:
        assert c[0, 0] == np.inf and c[0, 1] == np.inf


@pytest.mark.parametrize("n", [5, 40])
def test_infinitely_distant_pairs_add_nothing(n):
    """Without bonded terms: the energy is that of the ligand without the pairs of that atom."""
    lig = S.make_ligand(n, seed=n)
    lig = dataclasses.replace(lig, bond_k=0 * lig.bond_k, angles=np.zeros((0, 3), np.int32), angle_k=np.zeros(0),
                              angle_theta0=np.zeros(0), torsions=np.zeros((0, 4), np.int32),
                              torsion_V=np.zeros((0, 3)), torsion_gamma=np.zeros((0, 3)))
    # an atom of one bond; the ligand's other bonds, so that exclusions stay as they are
    last = next(a for a in range(n - 1, 0, -1) if (lig.bonds == a).sum() == 1)
    keep = ~(lig.bonds == last).any(1)
    cut = dataclasses.replace(lig, bonds=lig.bonds[keep], bond_k=lig.bond_k[keep], bond_r0=lig.bond_r0[keep])
    far = lig.x0[None].copy()
    far[0, last, 0] = np.inf
    gone = lig.x0[None].copy()
    gone[0, last, 0] = 1e18  # its pairs are below 1e-13 kcal/mol
    got, want = _evaluate(cut, far), _evaluate(cut, gone)
    for a, b in ((got[0], want[0]), (got[2], want[2])):
        assert np.isclose(a[0, 0], b[0, 0], rtol=1e-12, atol=1e-11)


def test_restraint_of_a_centre_that_is_not_a_number():
    lig = S.one_atom_ligand()
    x = np.array([[[0.5, np.nan, 0.25]]])
    c, F, _ = _evaluate(lig, x)
    assert np.isnan(c[0, 1]) and np.isfinite(F).all()


def _torsion_only():
    """A four-atom chain with its torsion alone."""
    n = 4
    return S.Ligand(mass=np.full(n, 12.0), charge=np.zeros(n), rstar=np.full(n, 1.8), eps=np.zeros(n),
                    bonds=np.array([[0, 1], [1, 2], [2, 3]], np.int32), bond_k=np.zeros(3), bond_r0=np.full(3, 1.4),
                    angles=np.zeros((0, 3), np.int32), angle_k=np.zeros(0), angle_theta0=np.zeros(0),
                    torsions=np.array([[0, 1, 2, 3]], np.int32), torsion_V=np.array([[1.0, 0.5, 0.25]]),
                    torsion_gamma=np.array([[0.0, np.pi, 0.0]]), x0=np.zeros((n, 3)))


@pytest.mark.parametrize("scale", [1e-15, 1.0, 1e20, 1e37, 2.2e38])
def test_torsion_angle_at_any_scale(scale):
    """The angle does not depend on the scale, also where products of four lengths leave the range of a double's
    square (positions near 1e38 A)."""
    chain = np.array([[0.5, 1.0, 0.25], [0.0, 0.0, 0.0], [1.0, 0.25, 0.0], [1.25, 0.5, 1.5]])
    c, F, e = _evaluate(_torsion_only(), scale * np.repeat(chain[None], 3, 0))
    ref = _evaluate(_torsion_only(), chain[None])[0][0, 0]
    x = (scale * chain).astype(np.float32).astype(np.longdouble) / np.longdouble(scale)  # as rounded
    b1, b2, b3 = np.diff(x, axis=0)
    n1, n2 = np.cross(b1, b2), np.cross(b2, b3)
    phi = np.arctan2(np.sqrt(b2 @ b2) * (b1 @ n2), n1 @ n2)
    want = sum(v / 2 * (1 + np.cos(m * phi - g)) for m, v, g in ((1, 1.0, 0.0), (2, 0.5, np.pi), (3, 0.25, 0.0)))
    assert np.allclose(c[:, 0], float(want), rtol=1e-12) and np.allclose(e[:, 0], float(want), rtol=1e-12)
    assert abs(float(want) - ref) < 1e-5


def test_torsion_of_a_position_that_is_not_a_number():
    x = np.array([[[0.5, 1.0, 0.25], [0.0, 0.0, 0.0], [1.0, 0.25, 0.0], [1.25, np.nan, 1.5]]])
    c, F, e = _evaluate(_torsion_only(), x)
    assert np.isnan(c[0, 0]) and np.isnan(e[0, 0])
