"""Contexts beside each other: a kernel's shared-memory limit is one per device, so what one context loads or
lays out must not change what another's launches may ask for."""
import threading

import numpy as np
import pytest

import oracle
from paper_1507_03703_gb300 import synthetic as S

from systems import configurations, gpu_context, raw_grids32, state_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def small():
    sys_ = S.config_small(1)
    return sys_, raw_grids32(sys_), state_table(sys_)


@pytest.mark.parametrize("n_large,n_small", [(31, 10), (48, 34), (96, 70)])
def test_a_second_batch_of_smaller_ligands(small, n_large, n_small):
    """The two batches take the same kernel; the second asks for less shared memory."""
    from paper_1507_03703_gb300.algdock import Context
    sys_, g32, (T, alpha, dt) = small
    K = len(T)
    states = torch.arange(K, dtype=torch.int32, device="cuda")

    def batch(n):
        lig = S.make_ligand(n, seed=n, min_sep=2.6)
        ctx = Context(0)
        ctx.grids_load(sys_.grid, *g32, vmax_e=oracle.soft_elec_cap(lig))
        ctx.states_set(T, alpha, dt)
        ctx.batch_load([lig], sys_.site)
        ctx.batch_layout(np.zeros(K, dtype=np.int32), n)
        return ctx, configurations(sys_, K, seed=n, jitter=0.02, ligand=lig)

    def trial(ctx, x):
        xd = torch.from_numpy(x).cuda()
        comps = torch.empty((K, 4), dtype=torch.float64, device="cuda")
        dH = torch.empty(K, dtype=torch.float64, device="cuda")
        ctx.batch_hmc_cycle(states, xd, comps, dH, n_steps=2, seed=3, cycle=1)
        return xd.cpu().numpy(), comps.cpu().numpy(), dH.cpu().numpy()

    first, x = batch(n_large)
    before = trial(first, x)
    second, y = batch(n_small)
    assert second.batch_shapes() == first.batch_shapes()
    trial(second, y)
    for a, b in zip(before, trial(first, x)):
        assert np.array_equal(a, b, equal_nan=True)


def test_two_threads_with_ligands_of_different_size(small):
    """One context per thread; each thread's results are those it gets alone."""
    sys_, g32, (T, alpha, dt) = small
    n, K = 64, len(T)
    jobs = []
    for atoms in (46, 34):  # the same kernels, different shared memory
        lig = S.make_ligand(atoms, seed=atoms, min_sep=2.6)
        ctx = gpu_context(sys_, g32, T, alpha, dt, ligand=lig)
        stream = torch.cuda.Stream()
        ctx.set_stream(stream)
        x = torch.from_numpy(configurations(sys_, n, seed=atoms, jitter=0.02, ligand=lig)).cuda()
        sd = (torch.arange(n, device="cuda") % K).to(torch.int32)
        jobs.append((ctx, stream, x, sd, [torch.empty((n, 4), dtype=torch.float64, device="cuda") for _ in range(3)],
                     torch.empty_like(x), torch.empty_like(x)))
    torch.cuda.synchronize()
    errors = []

    def calls(job, count):
        ctx, stream, x, sd, comps, y, F = job
        try:
            for _ in range(count):
                with torch.cuda.stream(stream):
                    y.copy_(x)
                ctx.hmc_cycle(sd, y, comps[0], n_steps=1, seed=5, cycle=2)
                ctx.reduced_energies(n, x=x, comps=comps[1])
                ctx.energy_force(sd, x, F, comps[2])
        except Exception as e:  # noqa: BLE001 - reported by the test
            errors.append(e)

    def results(job):
        torch.cuda.synchronize()
        return [t.cpu().numpy() for t in (*job[4], job[5], job[6])]

    alone = []
    for job in jobs:
        calls(job, 1)
        alone.append(results(job))
    threads = [threading.Thread(target=calls, args=(job, 300)) for job in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
    for job, want in zip(jobs, alone):
        for a, b in zip(results(job), want):
            assert np.array_equal(a, b)
