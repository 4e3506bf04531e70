"""What an FP64 MBAR solve leaves allocated: the scratch of a large solve (1.2 GB of stored weights) is given
back when the call returns, that of a small one stays with its context and goes with it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_large_scratch_is_given_back():
    from paper_1507_03703_gb300.algdock import Context
    K, per = 256, 2400
    g = torch.Generator(device="cuda").manual_seed(1)
    beta = 0.5 ** (torch.arange(K, device="cuda", dtype=torch.float64) / (K - 1))
    u = torch.outer(beta, 30.0 + torch.rand(K * per, dtype=torch.float64, device="cuda", generator=g))
    N_k = np.full(K, per, dtype=np.int64)
    small_k = np.full(4, per, dtype=np.int64)
    small = u[:4, :4 * per].contiguous()
    ctx = Context(0)
    ctx.mbar(small, small_k, max_iter=2, raise_on_nonconvergence=False)  # modules and kernels are loaded
    before = _free()
    first, _ = ctx.mbar(u, N_k, max_iter=4, raise_on_nonconvergence=False)
    assert before - _free() < 64 << 20
    again, _ = ctx.mbar(u, N_k, max_iter=4, raise_on_nonconvergence=False)
    assert np.array_equal(first, again)
    del ctx
    assert before - _free() < 64 << 20
