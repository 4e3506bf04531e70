"""The log-sum-exp passes of MBAR at their edges: state counts around the loads in flight and the tile
of 256, sample counts around the blocks and chunks, unsampled states, infinite reduced energies.

Three iterations against the same in 64-bit torch.  Bound of the FP32 modes: an exponential is within
2^-21 relative and an argument (below 64 here wherever it counts) within 64 * 2^-24, so 4.3e-6 a pass, two
passes an iteration, the gauge doubles, three iterations: 5.2e-5.  FP64: 1e-11."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _iterate(u, N_k, iters):
    logN = torch.log(torch.as_tensor(N_k, device="cuda", dtype=torch.float64))
    f = torch.zeros(u.shape[0], dtype=torch.float64, device="cuda")
    for _ in range(iters):
        logD = torch.logsumexp((logN + f)[:, None] - u, 0)
        f = -torch.logsumexp(-u - logD, 1)
        f = f - f[0].clone()
    return f.cpu().numpy()


@pytest.mark.parametrize("K,N", [(1, 1), (2, 33), (7, 255), (16, 4097), (17, 12289), (40, 8193), (257, 515), (300, 9001)])
@pytest.mark.parametrize("edges", [False, True])
def test_three_iterations(K, N, edges):
    from paper_1507_03703_gb300.algdock import Context
    rng = np.random.default_rng(1000 * K + N)
    # harmonic wells over a common interval, in rising and falling order of their energies
    centre = rng.uniform(-1.5, 1.5, size=K)
    x = rng.normal(size=N)
    u = 0.5 * rng.uniform(0.5, 4.0, size=(K, 1)) * (x[None] - centre[:, None]) ** 2 + rng.uniform(-3, 3, size=(K, 1))
    u += 5.0 * rng.random(N)[None]
    N_k = np.full(K, N // K, dtype=np.int64)
    N_k[0] += N - N_k.sum()
    if edges and K > 2:
        N_k[0] += N_k[2]
        N_k[2] = 0
        u[1, ::97] = np.inf
    ud = torch.from_numpy(u).cuda()
    want = _iterate(ud, N_k, 3)
    ctx = Context(0)
    for mode, bound in ((0, 1e-11), (1, 5.2e-5), (2, 5.2e-5)):
        f, _ = ctx.mbar(ud, N_k, tol=1e-300, max_iter=3, precision_mode=mode, raise_on_nonconvergence=False)
        assert np.abs(f - want).max() <= bound, (mode, np.abs(f - want).max())
