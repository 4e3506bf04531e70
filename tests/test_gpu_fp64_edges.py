"""The all-FP64 path at the edges of its warp layout, against the FP64 oracle: atom counts around the
32 lanes and both parities of the pair ring, configuration counts around a block, no forces wanted,
and topologies whose bonded slots leave room for one configuration per block or for none.  Bounds as
in test_gpu_fp64.py: both sides are FP64 and differ in the order of sums and in the maths library,
1e-10 relative."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1507_03703_gb300 import synthetic as S

from systems import configurations, state_table
from test_gpu_fp64 import _arms, _check

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def small():
    sys_ = S.config_small(1)
    return sys_, oracle.grid_direct_sum(sys_.receptor, sys_.grid), state_table(sys_)


@pytest.mark.parametrize("n_atoms,n", [(2, 1), (3, 2), (4, 3), (16, 4), (31, 5), (32, 7), (34, 9), (64, 3), (65, 6),
                                       (95, 2)])
def test_atom_and_configuration_counts(small, n_atoms, n):
    sys_, raw64, (T, alpha, dt) = small
    lig = S.make_ligand(n_atoms, seed=n_atoms, min_sep=2.6)
    ctx, osys = _arms(sys_, lig, T, alpha, dt, raw64)
    x = configurations(sys_, n, seed=6, jitter=0.1, ligand=lig)
    _check(ctx, osys, x, (np.arange(n) * 5) % len(T))


@pytest.mark.parametrize("copies", [150, 300])
def test_many_bonded_terms(small, copies):
    """A 20-atom tree whose bonds count `copies` times (19 * copies * 2 slots and the rest): 5,700 of
    them leave one configuration per block, 11,400 none."""
    sys_, raw64, (T, alpha, dt) = small
    base = sys_.ligand
    lig = dataclasses.replace(base, bonds=np.tile(base.bonds, (copies, 1)), bond_k=np.tile(base.bond_k, copies) / copies,
                              bond_r0=np.tile(base.bond_r0, copies))
    ctx, osys = _arms(sys_, lig, T, alpha, dt, raw64)
    x = configurations(sys_, 3, seed=7, jitter=0.1, ligand=lig)
    _check(ctx, osys, x, np.array([0, 9, 15]))
