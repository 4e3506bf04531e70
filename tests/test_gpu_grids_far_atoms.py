"""algdock_grids_build with receptor atoms (and lattice nodes) farther away than FP32 coordinates reach: their
terms vanish, as in FP64.  Reference and bounds of test_gpu_grids_build_edges.py; a term below the smallest
normal float (1.2e-38, times the Coulomb constant and a charge) may round to zero or to that."""
import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

from test_gpu_grids_build_edges import U, _receptor, _reference

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _check(rec, grid):
    from paper_1507_03703_gb300.algdock import Context
    shape = (grid.n[2], grid.n[1], grid.n[0])
    out = [torch.full(shape, np.nan, dtype=torch.float32, device="cuda") for _ in range(3)]
    Context(0).grids_build(grid, rec, *out)
    with np.errstate(over="ignore"):  # a squared distance beyond FP64 is infinite, its terms zero
        want = _reference(rec, grid)
    for got, (w, mag), bound in zip(out, want, (49 * U, 25 * U, 9 * U)):
        err = np.abs(got.cpu().numpy().astype(np.float64).ravel() - w)
        assert np.all(err <= bound * mag + 1e-34)


@pytest.mark.parametrize("far", [1e12, 1e15, 1e17, 3e18, 1e19, 3e19, 1e25, 4e38, 1e120, -1e300])
@pytest.mark.parametrize("spacing", [0.25, 0.3])
def test_far_atoms(far, spacing):
    grid = S.GridSpec(origin=np.array([-1.0, 0.5, 0.25]), spacing=spacing, n=(9, 4, 3))
    rec = _receptor(5, 3)
    rec.xyz[1] = [far, 0.0, 1.0]
    rec.xyz[4] = [-1.0, -far, 0.5 * far]
    _check(rec, grid)
    alone = S.Receptor(xyz=rec.xyz[1:2], rstar=rec.rstar[1:2], eps=rec.eps[1:2], charge=rec.charge[1:2])
    _check(alone, grid)


@pytest.mark.parametrize("spacing", [1e6, 1e18, 7e19, 1e200])
def test_far_nodes(spacing):
    rec = _receptor(4, 5)
    rec.xyz[2] = [1e250, 0.0, 0.0]
    _check(rec, S.GridSpec(origin=np.zeros(3), spacing=spacing, n=(6, 2, 3)))
