"""The error of algdock_grids_build against 64 bits is no larger than that of FP32 terms of FP64 differences
with IEEE divisions, summed in FP64.

Root-mean-square of the error over a node's sum of magnitudes, over receptors and lattices; the geometric mean of
the ratios of the two over them is at most 1.005 (the rounding of single terms moves one lattice's ratio by up
to a per cent either way)."""
import numpy as np
import pytest

from paper_1507_03703_gb300 import synthetic as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LATTICES = [(25, 0.25, 300), (33, 0.5, 1500), (41, 0.375, 800), (49, 0.25, 900), (45, 0.5, 600)]


def _sums(nodes, rec, terms):
    """Per node the FP64 sums and sums of magnitudes of the three channels' terms, by chunks."""
    dev = nodes.device
    pos = torch.as_tensor(rec, device=dev)
    parts = [terms(nodes[b:b + 2048, None] - pos[None]) for b in range(0, len(nodes), 2048)]
    return [torch.cat([p[c].double().sum(-1) for p in parts]) for c in range(3)], \
        [torch.cat([p[c].double().abs().sum(-1) for p in parts]) for c in range(3)]


def _errors(n, h, n_rec, seed):
    from paper_1507_03703_gb300.algdock import Context
    rec, grid = S.make_receptor(n_rec, np.zeros(3), seed), S.cube_grid(np.zeros(3), h, n)
    out = [torch.empty((n,) * 3, dtype=torch.float32, device="cuda") for _ in range(3)]
    Context(0).grids_build(grid, rec, *out)
    ax = h * torch.arange(n, dtype=torch.float64, device="cuda")
    z, y, x = torch.meshgrid(ax, ax, ax, indexing="ij")
    nodes = torch.stack([x, y, z], -1).reshape(-1, 3)
    pos = rec.xyz - grid.origin
    two_r, eps = (torch.as_tensor(v, device="cuda") for v in (2.0 * rec.rstar, rec.eps))
    A, B = eps.sqrt() * two_r ** 6, (2.0 * eps).sqrt() * two_r ** 3
    Q = torch.as_tensor(rec.charge / 4.0, device="cuda")

    def exact(d):
        r2 = (d * d).sum(-1)
        i2, a2 = 1.0 / r2.clamp(min=1e-4), 1.0 / r2.clamp(min=4.0)
        return A * i2 ** 6, -B * a2 ** 3, 332.0637 * Q * a2

    def fp32(d):
        def fma(a, b, c):  # the product of two floats is exact in FP64
            return (a.double() * b.double() + c.double()).float()
        dx, dy, dz = d.float().unbind(-1)
        r2 = fma(dz, dz, fma(dy, dy, dx * dx))
        i2, a2 = 1.0 / r2.clamp(min=1e-4), 1.0 / r2.clamp(min=4.0)
        i6 = (i2 * i2) * i2
        return A.float() * (i6 * i6), -B.float() * ((a2 * a2) * a2), Q.float() * a2

    want, mag = _sums(nodes, pos, exact)
    plain, _ = _sums(nodes, pos, fp32)
    plain = [plain[0].float(), plain[1].float(), (332.0637 * plain[2]).float()]
    rms = lambda got: [float((((g.double().ravel() - w) / m) ** 2).mean().sqrt()) for g, w, m in zip(got, want, mag)]
    return np.array(rms(out)) / np.array(rms(plain))


def test_error_against_64_bits():
    ratios = np.array([_errors(n, h, n_rec, seed) for n, h, n_rec in LATTICES for seed in (1, 2, 3)])
    assert np.all(np.exp(np.log(ratios).mean(0)) <= 1.005), np.exp(np.log(ratios).mean(0))
