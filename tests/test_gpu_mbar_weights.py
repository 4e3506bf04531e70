"""The FP64 mode of algdock_mbar on stored weights against the oracle's log-sum-exp iteration: the
edges of its warps and tiles (states per warp, 32-sample tiles), ladders whose reduced energies
leave the range the weights are exact in, infinite energies, and the sizes that keep the
log-sum-exp kernels.  Bounds as for the log-sum-exp kernels (test_gpu_mbar.py): both sides sum the
same terms in FP64, so f agrees within 1e-8 kT at a 1e-10 tolerance, and the iteration counts within
one (the stopping test compares a change near the tolerance)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    from paper_1507_03703_gb300.algdock import Context
    return Context(0)


def _ladder(K, N_k, seed, dof=40.0, scale=0.5, offset=0.0):
    """Reduced energies beta_k E of gamma-distributed E sampled at each beta, with an offset per
    sample that cancels in MBAR."""
    rng = np.random.default_rng(seed)
    beta = scale ** (np.arange(K) / max(K - 1, 1))
    E = np.concatenate([rng.gamma(dof, 1.0 / b, size=n) for b, n in zip(beta, N_k)])
    return beta[:, None] * E[None, :] + offset * rng.normal(size=E.size)[None, :]


def _check(ctx, u, N_k, tol=1e-10):
    f_o, it_o = oracle.mbar(u, N_k, tol=tol)
    f, it = ctx.mbar(torch.from_numpy(u).cuda(), N_k, tol=tol)
    assert np.max(np.abs(f - f_o)) < 1e-8
    assert abs(it - it_o) <= 1


@pytest.mark.parametrize("K,per", [(1, 5), (2, 16), (3, 11), (4, 8), (31, 7), (32, 1), (33, 9), (127, 3), (128, 5),
                                   (129, 3), (255, 2), (256, 3), (257, 2)])
def test_edges_of_warps_and_tiles(ctx, K, per):
    N_k = np.full(K, per, dtype=np.int64)
    N_k[-1] += 1  # uneven counts, and sample numbers on both sides of a multiple of 32
    _check(ctx, _ladder(K, N_k, seed=K), N_k)


def test_many_tiles_per_block(ctx):
    N_k = np.full(5, 9001, dtype=np.int64)
    _check(ctx, _ladder(5, N_k, seed=3), N_k)


@pytest.mark.parametrize("dof", [800.0, 3000.0])
def test_wide_ladder_takes_the_log_sum_exp_iteration_first(ctx, dof):
    """f spans dof ln 2 (555 and 2079 kT): from f = 0 the state sums lie below the limits."""
    K = 96
    N_k = np.full(K, 40, dtype=np.int64)
    _check(ctx, _ladder(K, N_k, seed=8, dof=dof, offset=50.0), N_k)


def test_infinite_energies_have_no_weight(ctx):
    K = 6
    N_k = np.full(K, 50, dtype=np.int64)
    u = _ladder(K, N_k, seed=4)
    u[4, ::3] = np.inf
    u[:3, 1::7] = np.inf
    _check(ctx, u, N_k)


def test_nan_does_not_converge(ctx):
    N_k = np.full(3, 20, dtype=np.int64)
    u = _ladder(3, N_k, seed=5)
    u[1, 7] = np.nan
    _, it = ctx.mbar(torch.from_numpy(u).cuda(), N_k, max_iter=40, raise_on_nonconvergence=False)
    assert it == -1
