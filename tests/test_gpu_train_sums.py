"""Gradients from the forward's per-point sums against FP64 autograd over the
neighbour lists of a debug call: shared-memory and spilled leaves, other kernel
exponents, a large epsilon, the kNN within P_2 and the cross-leaf neighbours.

Tolerance: a term's FP32 factors (exponential, quotient, logarithm) are each good
to a few ulp, 1e-6 relative together; the sums carry no further rounding that
counts, so a gradient is within 2e-6 of the sum of its terms' magnitudes."""

import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cloud(n):
    g = torch.Generator().manual_seed(n)
    v = torch.randn(n - n // 10, 3, generator=g)
    surf = v / v.norm(dim=1, keepdim=True) + 0.005 * torch.randn(n - n // 10, 3, generator=g)
    return torch.cat([surf, 2.4 * torch.rand(n // 10, 3, generator=g) - 1.2]).cuda()


@pytest.mark.parametrize("n,kw", [
    (9000, {"k": 16}), (9000, {"k": 9, "gamma": 3.0, "eps_k": 1e-2, "sigma": 0.7, "alpha": -0.5}),
    (3000, {"k": 12, "leaf_capacity": 0xFFFFFFFF}), (9000, {"k": 16, "rescore_p2": 1}),
    (9000, {"k": 16, "cross_leaf": 1, "leaf_capacity": 128}), (30_000, {"k": 64, "leaf_capacity": 512}),
])
def test_gradient_against_autograd(n, kw):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    xyz = _cloud(n)
    P = Params(**{"alpha": 1.3, "sigma": 0.9, "gamma": 2.0, "select_mode": 1, "tau": 7.0, "temperature": 0.7,
                  "eps_k": 1e-9, **kw})
    d = Denoiser(max_points=n)
    try:
        if P.cross_leaf:
            d.set_cross_leaf(True)
        g = d.run_debug(xyz, P)
        d.set_training(True)
        d.run(xyz, P)
        r = d.soft_removal(n)
        u = torch.randn(n, generator=torch.Generator().manual_seed(1)).cuda()
        got = d.backward(u)
    finally:
        d.close()
    scored = ((g["stage"] == 0) | (g["stage"] == 3)) & (g["score"] > 0)
    i = torch.nonzero(scored).flatten()
    nbr = g["nbr"][i].long()
    ok = nbr >= 0
    nbr = nbr.clamp(min=0)
    d2 = g["nbr_d2"][i].double()
    r2 = g["r2"].double()
    keff = (g["nbr"] >= 0).sum(1).double()
    rho = keff / (4 / 3 * math.pi * r2 ** 1.5)
    ref = (g["leaf_rho_med"] ** 2 + P.eps_rho).sqrt()[i]
    lw = torch.log(rho[nbr] / ref[:, None]) + torch.log(rho[i] / ref)[:, None]
    th = torch.tensor([P.alpha, P.sigma, P.gamma, P.tau], dtype=torch.float64, device="cuda", requires_grad=True)
    base = torch.where(ok, d2, 1.0)
    D = base ** (th[2] / 2)
    t = torch.where(ok, torch.exp(0.5 * th[0] * lw - base / (2 * th[1] ** 2 * r2[i][:, None])) / (D + P.eps_k), 0.0)
    F = t.sum(1)
    rr = 1 - torch.sigmoid((torch.log(F) - th[3]) / P.temperature)
    assert torch.allclose(rr.detach(), r[i].double(), rtol=1e-4, atol=1e-6)
    (rr * u[i].double()).sum().backward()
    m = 1 - rr.detach()
    w = (u[i].double() * m * (1 - m) / P.temperature / F.detach()).abs()
    t = t.detach()
    mag = [(w * (t * 0.5 * lw.abs().nan_to_num(0, 0, 0)).sum(1)).sum(),
           (w * (t * base / (P.sigma ** 3 * r2[i][:, None])).sum(1)).sum(),
           (w * (t * 0.5 * torch.log(base).abs()).sum(1)).sum(), (w * F.detach()).sum()]
    # (m itself is FP32 through ln F: m (1 - m) is good to |ln F| * 2^-23 / T, below 1e-5)
    for q in range(4):
        assert abs(got[q] - th.grad[q].item()) <= 2e-5 * mag[q].item(), (q, got[q], th.grad[q].item(), mag[q].item())
