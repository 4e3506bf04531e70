"""Learned moves in one call against the same moves one call at a time, bit for bit: the network's
outputs at the current pose are kept between the moves of a call and replaced where a move was
accepted.  And the fused forward pass on either side of its two row-tile sizes: a row's outputs do not
depend on how many rows there are."""
import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

from systems import configurations, gpu_context, raw_grids32, state_table

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def small():
    sys_ = S.config_small(1)
    T, alpha, dt = state_table(sys_)
    return sys_, gpu_context(sys_, raw_grids32(sys_), T, alpha, dt), len(T)


@pytest.mark.parametrize("n", [1, 6, 2433])
def test_moves_in_one_call_equal_single_moves(small, n):
    from paper_1507_03703_gb300.learned import LearnedProposal
    sys_, ctx, K = small
    lp = LearnedProposal(ctx, seed=4, n_torsions=0)
    x0 = torch.from_numpy(configurations(sys_, 32, seed=3, jitter=0.02)[np.arange(n) % 32]).cuda()
    st = torch.from_numpy((K // 2 + np.arange(n) % 3).astype(np.int32)).cuda()
    st[n // 2] = -1 if n > 1 else st[0]
    c0 = torch.zeros((n, 4), dtype=torch.float64, device="cuda")
    ctx.reduced_energies(n, x=x0, comps=c0)
    got = []
    for calls in (1, 3):
        x, c = x0.clone(), c0.clone()
        acc = torch.zeros(n, dtype=torch.int32, device="cuda")
        for k in range(calls):
            lp.propose(st, x, c, 3 // calls, seed=9, cycle=5 if calls == 1 else 15 + k, accepted=acc)
        got.append((x, c, acc))
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert n < 100 or got[0][2].sum() > 0


def test_forward_rows_do_not_depend_on_the_row_count(small):
    from paper_1507_03703_gb300.algdock import MLP_NFEAT, pack_mlp
    _, ctx, _ = small
    flat, w = pack_mlp(S.mlp_init(2))
    params, wb = torch.from_numpy(flat).cuda(), torch.from_numpy(w.view(np.int16)).cuda()
    feat = torch.randn((2465, MLP_NFEAT), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    full = torch.empty((2465, 360), device="cuda")
    ctx.mlp_forward(params, wb, feat, full)
    for a, b in ((0, 1), (0, 17), (2432, 2465), (0, 2432), (32, 2465)):
        out = torch.empty((b - a, 360), device="cuda")
        ctx.mlp_forward(params, wb, feat[a:b].contiguous(), out)
        assert torch.equal(out, full[a:b])
