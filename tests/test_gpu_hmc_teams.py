"""The HMC trial by teams of warps: every launch shape (one replica per team, spread over the SMs; once
and twice around; from the work counter) against the same replicas launched in other numbers, bit for
bit: a replica's arithmetic does not depend on how it was launched.  One, two and three warps per
team, with and without the pair table, even and odd atom counts, full and split last pair passes.
(The comparison with the oracle over atom counts is in test_gpu_hmc.py, test_gpu_edges.py and
test_gpu_batch.py.)"""
import dataclasses

import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

from systems import configurations, gpu_context, raw_grids32, state_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def small():
    sys_ = S.config_small(1)
    return sys_, raw_grids32(sys_), state_table(sys_)


def _trial(ctx, x, states, n_steps, rep_offset=0):
    xd, sd = torch.from_numpy(x.copy()).cuda(), torch.from_numpy(states).cuda()
    n = x.shape[0]
    comps = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    dH = torch.zeros(n, dtype=torch.float64, device="cuda")
    acc = torch.zeros(n, dtype=torch.uint8, device="cuda")
    cnt = torch.zeros(4, dtype=torch.int64, device="cuda")
    ctx.hmc_cycle(sd, xd, comps, dH, acc, n_steps=n_steps, seed=11, cycle=2, rep_offset=rep_offset, counters=cnt)
    return [t.cpu().numpy() for t in (xd, comps, dH, acc, cnt)]


@pytest.mark.parametrize("n_atoms,bonds", [(20, 1), (32, 1), (47, 1), (48, 1), (48, 30), (61, 30), (70, 1), (83, 1),
                                           (96, 1)])
def test_launch_shapes_give_the_same_bits(small, n_atoms, bonds):
    """bonds > 1 repeats the bonds so often that the ligand's pair table no longer fits."""
    sys_, g32, (T, alpha, dt) = small
    lig = S.make_ligand(n_atoms, seed=n_atoms, min_sep=2.6)
    lig = dataclasses.replace(lig, bonds=np.tile(lig.bonds, (bonds, 1)), bond_k=np.tile(lig.bond_k, bonds) / bonds,
                              bond_r0=np.tile(lig.bond_r0, bonds))
    ctx = gpu_context(sys_, g32, T, alpha, dt, ligand=lig)
    assert ctx.hmc_shape()[1] == (n_atoms <= 48 and bonds == 1)
    n = 5000
    x = configurations(sys_, 64, seed=10, jitter=0.02, ligand=lig)[np.arange(n) % 64]
    states = (np.arange(n) * 5 % len(T)).astype(np.int32)
    states[7] = -1  # an invalid state leaves its replica untouched
    whole = _trial(ctx, x, states, 2)
    assert np.isnan(whole[2][7]) and np.array_equal(whole[0][7], x[7])
    for count in (1, 17, 153, 700, 1500, 2500):
        part = _trial(ctx, x[:count], states[:count], 2)
        for a, b in zip(part[:4], whole[:4]):
            assert np.array_equal(a, b[:count], equal_nan=a.dtype.kind == "f"), count
    tail = _trial(ctx, x[4990:], states[4990:], 2, rep_offset=4990)
    for a, b in zip(tail[:4], whole[:4]):
        assert np.array_equal(a, b[4990:], equal_nan=a.dtype.kind == "f")
