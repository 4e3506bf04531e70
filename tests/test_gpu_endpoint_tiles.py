"""The target interaction at sizes that take the block shapes test_gpu_endpoint_shapes.py does not reach: four
points a thread, and groups of threads that have no receptor tile in a round.  Bounds as there."""
import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

from test_gpu_endpoints import _check_psi, _ctx

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_atoms,n_rec,N", [
    (61, 257, 3001),  # four points a thread, one pair in the second tile, a ragged last block
    (70, 513, 5003),  # four points a thread, three tiles
    (33, 129, 6001),  # four points a thread, half a tile
    (33, 257, 1501),  # two groups of three points, one pair in the second group's tile
    (13, 513, 2000),  # four groups of three points, the last without a tile
    (2, 515, 300),    # four groups of one point, the last without a tile
    (10, 200, 500),   # two groups of one point, the second without a tile
])
def test_tiles(n_atoms, n_rec, N):
    lig = S.make_ligand(n_atoms, seed=n_atoms)
    rec = S.make_receptor(n_rec, np.zeros(3), seed=5)
    ctx = _ctx(S.System(ligand=lig, receptor=rec, grid=S.cube_grid(np.zeros(3), 0.5, 9), site=np.zeros(3), legs=[]))
    rng = np.random.default_rng(n_rec)
    x = (lig.x0[None] + rng.normal(scale=1.0, size=(N, 1, 3))).astype(np.float32)
    got = ctx.target_interaction(torch.from_numpy(x).cuda()).cpu().numpy()
    pick = np.unique(np.concatenate([np.arange(12), np.arange(N - 12, N), rng.integers(0, N, 40)]))
    _check_psi(rec, lig, x[pick], got[pick])
