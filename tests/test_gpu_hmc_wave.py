"""The HMC launch of two-warp teams around the replica counts that one block of 16 teams per SM takes at
once, against the same replicas in launches on either side, bit for bit."""
import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

from systems import configurations, gpu_context
from test_gpu_hmc_teams import _trial, small  # noqa: F401

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


@pytest.mark.parametrize("n_atoms", [33, 47, 48])
def test_one_wave_of_sixteen(small, n_atoms):  # noqa: F811
    sys_, g32, (T, alpha, dt) = small
    lig = S.make_ligand(n_atoms, seed=n_atoms, min_sep=2.6)
    ctx = gpu_context(sys_, g32, T, alpha, dt, ligand=lig)
    n = 4000
    x = configurations(sys_, 64, seed=10, jitter=0.02, ligand=lig)[np.arange(n) % 64]
    states = (np.arange(n) * 5 % len(T)).astype(np.int32)
    states[7] = -1
    whole = _trial(ctx, x, states, 2)
    for count in (1824, 1825, 2000, 2432, 2433):
        part = _trial(ctx, x[:count], states[:count], 2)
        for a, b in zip(part[:4], whole[:4]):
            assert np.array_equal(a, b[:count], equal_nan=a.dtype.kind == "f"), count
