"""The block shapes of the target interaction and the merge of the FEP sums at their edges.

Bounds as in test_gpu_endpoints: 2e-5 of the sum of the terms' magnitudes for a configuration's
energy (FP32 terms, FP32 sums of a tile, FP64 sums of tiles), 1e-12 relative for the FP64 sums."""
import math

import numpy as np
import pytest

import oracle
from paper_1507_03703_gb300 import synthetic as S

from test_gpu_endpoints import _check_psi, _ctx, _fep_close

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_atoms,n_rec,N", [
    (96, 700, 1),      # one configuration: two groups of one point a thread, an odd last round
    (64, 1023, 150),   # a block per configuration, an odd receptor
    (10, 300, 500),    # one point a thread, a group with no tile in the last round
    (13, 1100, 2000),  # four groups
    (33, 257, 3001),   # one group, three points a thread, one pair in the last tile
    (61, 130, 5003),   # four points a thread, a ragged last block
])
def test_block_shapes(n_atoms, n_rec, N):
    lig = S.make_ligand(n_atoms, seed=n_atoms)
    rec = S.make_receptor(n_rec, np.zeros(3), seed=5)
    sys_ = S.System(ligand=lig, receptor=rec, grid=S.cube_grid(np.zeros(3), 0.5, 9), site=np.zeros(3), legs=[])
    ctx = _ctx(sys_)
    rng = np.random.default_rng(n_rec)
    x = (lig.x0[None] + rng.normal(scale=1.0, size=(N, 1, 3))).astype(np.float32)
    got = ctx.target_interaction(torch.from_numpy(x).cuda())
    assert torch.equal(got, ctx.target_interaction(torch.from_numpy(x).cuda()))
    pick = np.unique(np.concatenate([np.arange(min(N, 12)), np.arange(max(0, N - 12), N),
                                     rng.integers(0, N, 40)]))
    _check_psi(rec, lig, x[pick], got.cpu().numpy()[pick])


@pytest.mark.parametrize("N", [1, 33, 257, 4097, 80_001])
def test_fep_smallest_anywhere(N):
    """The smallest difference in the first, a middle and the last sample, far below the others (their
    weights vanish) and close to them, with weightless samples between."""
    ctx = _ctx(S.config_small(1))
    rng = np.random.default_rng(N)
    for at in sorted({0, N // 2, N - 1}):
        for low in (-900.0, -2.0):
            du = rng.normal(3.0, 2.0, size=N)
            du[rng.random(N) < 0.1] = np.inf
            du[at] = low
            _fep_close(ctx.fep(torch.from_numpy(du).cuda()), oracle.fep(du))
    g = ctx.fep(torch.full((N,), math.inf, dtype=torch.float64, device="cuda"))
    assert g["f"] == math.inf and g["n_eff"] == 0.0 and math.isnan(g["sigma"]) and g["du_min"] == math.inf
