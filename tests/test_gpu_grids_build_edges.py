"""algdock_grids_build against FP64 direct sums in numpy: lattices at the edges of a thread's four
nodes and of the receptor slices, spacings with and without a low part in the node coordinates, odd
and empty receptors, an atom on a node, atoms far outside the lattice.

Bounds, in units of u = 2^-24 relative to the sum of the terms' magnitudes: a difference carries one
rounding (and its low part one more), r^2 two of those and two of its own sums (6u), the reciprocal
one more (7u); r^-6 then 23u, r^-12 47u; a factor and the stored result add one each."""
import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
U = 2.0 ** -24


def _reference(rec, grid):
    ax = [grid.spacing * np.arange(grid.n[d]) for d in range(3)]
    z, y, x = np.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    nodes = np.stack([x, y, z], -1).reshape(-1, 3)
    d = nodes[:, None, :] - (rec.xyz - grid.origin)[None]
    r2 = (d * d).sum(-1)
    two_r = 2.0 * rec.rstar
    terms = [np.sqrt(rec.eps) * two_r ** 6 / np.maximum(r2, 1e-4) ** 6,
             -np.sqrt(2 * rec.eps) * two_r ** 3 / np.maximum(r2, 4.0) ** 3,
             332.0637 * 0.25 * rec.charge / np.maximum(r2, 4.0)]
    return [(t.sum(-1), np.abs(t).sum(-1)) for t in terms]


def _check(rec, grid):
    from paper_1507_03703_gb300.algdock import Context
    shape = (grid.n[2], grid.n[1], grid.n[0])
    out = [torch.full(shape, np.nan, dtype=torch.float32, device="cuda") for _ in range(3)]
    Context(0).grids_build(grid, rec, *out)
    for got, (want, mag), bound in zip(out, _reference(rec, grid), (49 * U, 25 * U, 9 * U)):
        err = np.abs(got.cpu().numpy().astype(np.float64).ravel() - want)
        assert np.all(err <= bound * mag + 1e-37), (err / np.maximum(mag, 1e-300)).max() / U


def _receptor(n, seed):
    rng = np.random.default_rng(seed)
    return S.Receptor(xyz=rng.uniform(-6.0, 9.0, size=(n, 3)), rstar=rng.uniform(1.5, 2.0, n),
                      eps=rng.uniform(0.01, 0.2, n), charge=rng.normal(0.0, 0.3, n))


@pytest.mark.parametrize("n", [(2, 3, 2), (4, 5, 3), (5, 2, 7), (9, 8, 33)])
@pytest.mark.parametrize("spacing", [0.25, 0.3])
@pytest.mark.parametrize("n_rec", [0, 1, 2, 255, 257, 601])
def test_lattice_edges(n, spacing, n_rec):
    _check(_receptor(n_rec, n_rec + n[0]), S.GridSpec(origin=np.array([-1.0, 0.5, 0.25]), spacing=spacing, n=n))


def test_one_slice_lattice():
    """Enough nodes that one thread sums the whole receptor for its four nodes."""
    _check(_receptor(21, 3), S.GridSpec(origin=np.array([-8.0, -8.0, -8.0]), spacing=0.2, n=(90, 84, 84)))


def test_atoms_on_nodes_and_far_away():
    rec = _receptor(40, 7)
    rec.xyz[0] = [0.0, 0.0, 0.0]          # a node
    rec.xyz[1] = [0.005, 0.0, 0.0]        # inside the floor of the repulsive sum
    rec.xyz[2] = [0.25 + 3e-5, 0.25, 0.5]
    rec.xyz[3] = [1e6, -2e5, 3.0]
    rec.xyz[4] = [1e20, 0.0, 0.0]         # r^2 overflows FP32
    _check(rec, S.GridSpec(origin=np.zeros(3), spacing=0.25, n=(6, 6, 6)))
