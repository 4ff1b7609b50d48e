"""dL/dgamma where eps_k is not small beside D = (d^2)^(gamma/2): its terms carry the
factor D / (D + eps_k), which must not be what is left of 1 after a subtraction.
Against FP64 over the neighbour lists of a debug call, for a few points at a time.

Tolerance: a term's FP32 factors (exponential, quotient, logarithm, (d^2)^(gamma/2)) and
m (1 - m) (FP32, through ln F) are good to 1e-5 of the term together, so the gradient
is within 2e-5 of the sum of its terms' magnitudes, the factor included."""

import math

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cloud(n, scale):
    g = torch.Generator().manual_seed(n)
    v = torch.randn(n - n // 10, 3, generator=g)
    surf = v / v.norm(dim=1, keepdim=True) + 0.005 * torch.randn(n - n // 10, 3, generator=g)
    return scale * torch.cat([surf, 2.4 * torch.rand(n // 10, 3, generator=g) - 1.2]).cuda()


@pytest.mark.parametrize("scale,kw", [
    (1.0, {"eps_k": 1e-12}), (1.0, {"eps_k": 1e-5}), (1.0, {"eps_k": 1e-3}), (0.03, {"eps_k": 1e-2}),
    (0.03, {"eps_k": 1.0}), (0.003, {"eps_k": 1.0}), (0.03, {"eps_k": 1e-2, "gamma": 3.0}),
    (0.03, {"eps_k": 1.0, "leaf_capacity": 0xFFFFFFFF}), (0.03, {"eps_k": 1.0, "cross_leaf": 1}), (1.0, {"eps_k": 0.0}),
])
def test_gamma_gradient(scale, kw):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    n = 5000
    xyz = _cloud(n, scale)
    P = Params(**{"k": 16, "select_mode": 1, "temperature": 0.7, "gamma": 2.0, **kw})
    d = Denoiser(max_points=n)
    try:
        if P.cross_leaf:
            d.set_cross_leaf(True)
        g = d.run_debug(xyz, P)
        i = torch.nonzero(((g["stage"] == 0) | (g["stage"] == 3)) & (g["score"] > 0)).flatten()
        P.tau = g["score"][i].log().median().item()  # (m near 1/2)
        d.set_training(True)
        d.run(xyz, P)
        picks = i[torch.randperm(len(i), generator=torch.Generator().manual_seed(3))[:12].cuda()]
        got = []
        for p in picks.tolist():
            u = torch.zeros(n, device="cuda")
            u[p] = 1.0
            got.append(d.backward(u)[2])
    finally:
        d.close()
    nbr = g["nbr"][picks].long()
    ok = nbr >= 0
    nbr = nbr.clamp(min=0)
    base = torch.where(ok, g["nbr_d2"][picks].double(), 1.0)
    r2 = g["r2"].double()
    rho = (g["nbr"] >= 0).sum(1).double() / (4 / 3 * math.pi * r2 ** 1.5)
    ref = (g["leaf_rho_med"] ** 2 + P.eps_rho).sqrt()[picks]
    lw = torch.log(rho[nbr] / ref[:, None]) + torch.log(rho[picks] / ref)[:, None]
    D = base ** (P.gamma / 2)
    t = torch.exp(0.5 * P.alpha * lw - base / (2 * P.sigma ** 2 * r2[picks][:, None])) / (D + P.eps_k)
    t = torch.where(ok, t, 0.0)
    F = t.sum(1)
    m = torch.sigmoid((torch.log(F) - P.tau) / P.temperature)
    w = m * (1 - m) / P.temperature / F
    term = t * 0.5 * torch.log(base) * D / (D + P.eps_k)
    want, mag = w * term.sum(1), w * term.abs().sum(1)
    err = (torch.tensor(got, dtype=torch.float64, device="cuda") - want).abs()
    assert (err <= 2e-5 * mag).all(), (err / mag).tolist()
