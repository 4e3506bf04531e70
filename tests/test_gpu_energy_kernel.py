"""The energies-only kernel of algdock_reduced_energies at the edges of its pair passes (full and split
last passes, odd partner ranges, odd atom counts) against the kernel of algdock_energy_force, which
takes one partner at a time: FP32 terms in the same order, so the bound of test_gpu_grids_energy.py
(1e-5 relative of a component plus 1e-4 kcal/mol) holds with room.  Few and many configurations (one
and four per warp) give the same bits, and u_kn formed with the energies equals u_kn formed from the
components."""
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


@pytest.mark.parametrize("n_atoms", [1, 2, 15, 16, 17, 31, 32, 33, 34, 35, 46, 47, 48, 49, 64, 65, 66, 67, 80, 81, 95, 96])
def test_components_match_the_force_kernel(small, n_atoms):
    sys_, g32, (T, alpha, dt) = small
    lig = S.one_atom_ligand() if n_atoms == 1 else S.make_ligand(n_atoms, seed=n_atoms, min_sep=2.6)
    ctx = gpu_context(sys_, g32, T, alpha, dt, ligand=lig)
    n = 37
    x = torch.from_numpy(configurations(sys_, n, seed=12, jitter=0.05, ligand=lig)).cuda()
    comps = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    ctx.reduced_energies(n, x=x, comps=comps)
    ref = torch.zeros_like(comps)
    force = torch.empty_like(x)
    ctx.energy_force(torch.zeros(n, dtype=torch.int32, device="cuda"), x, force, ref)
    a, b = comps.cpu().numpy(), ref.cpu().numpy()
    assert np.all(np.abs(a - b) <= 1e-5 * np.abs(b) + 1e-4)


@pytest.mark.parametrize("n_atoms", [20, 47, 70])
def test_tiles_and_fused_reduced_energies(small, n_atoms):
    sys_, g32, (T, alpha, dt) = small
    lig = S.make_ligand(n_atoms, seed=n_atoms, min_sep=2.6)
    ctx = gpu_context(sys_, g32, T, alpha, dt, ligand=lig)
    n, K = 60013, len(T)
    base = configurations(sys_, 101, seed=13, jitter=0.05, ligand=lig)
    x = torch.from_numpy(base[np.arange(n) % 101]).cuda()
    comps = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    u = torch.zeros((5, n), dtype=torch.float64, device="cuda")
    ctx.reduced_energies(n, x=x, comps=comps, k_begin=3, k_count=5, u_kn=u)
    few = torch.zeros((101, 4), dtype=torch.float64, device="cuda")
    ctx.reduced_energies(101, x=x, comps=few)
    assert torch.equal(comps, few[torch.arange(n, device="cuda") % 101])
    v = torch.zeros_like(u)
    ctx.reduced_energies(n, comps=comps, k_begin=3, k_count=5, u_kn=v)
    assert torch.equal(u, v)
    ctx.reduced_energies(n, x=x, k_begin=3, k_count=5, u_kn=v.zero_())  # no components wanted
    assert torch.equal(u, v)
