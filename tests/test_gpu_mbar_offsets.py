"""Large energies common to a sample's column cancel in MBAR's FP64 mode: a constant added to every reduced
energy of a sample leaves f as it was.

Reduced energies and constants are multiples of 2^-20 below 2^31, so every sum and difference of the first
iteration is exact, and f agrees with the solve without constants to rounding (1e-12) and that one with the
oracle within 1e-8 kT at a 1e-10 tolerance.  The constants put a column's largest log-weight `above` past the
next multiple of 2^-20 of itself, where exp(above) is near the largest double."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("above", [0.25, 700.0, 708.5, 709.5])
@pytest.mark.parametrize("K", [5, 140])
def test_a_sample_constant_cancels(K, above, sign):
    from paper_1507_03703_gb300.algdock import Context
    rng = np.random.default_rng(K)
    N_k = np.full(K, 40, dtype=np.int64)
    beta = 0.8 ** (np.arange(K) / (K - 1))
    E = np.concatenate([rng.gamma(40.0, 1.0 / b, size=n) for b, n in zip(beta, N_k)])
    u = np.round(beta[:, None] * E[None, :] * 2.0 ** 20) / 2.0 ** 20
    top = sign * (2.0 ** 30 + 1024.0 * rng.integers(0, 1000, E.size) + np.where(np.arange(E.size) % 3, 0.25, above))
    shifted = u - (u.min(0) + top)[None, :]
    assert np.array_equal(-shifted.min(0), top)
    ctx = Context(0)
    f0, it0 = ctx.mbar(torch.from_numpy(u).cuda(), N_k, precision_mode=0)
    f1, it1 = ctx.mbar(torch.from_numpy(shifted).cuda(), N_k, precision_mode=0)
    assert np.max(np.abs(f0 - oracle.mbar(u, N_k, tol=1e-10)[0])) < 1e-8
    assert np.max(np.abs(f1 - f0)) < 1e-12
    assert abs(it1 - it0) <= 1
