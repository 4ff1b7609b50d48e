"""The leaf kernel's CTA width, chosen from the number of points and the leaf
size, never changes a result: every width against 128-thread CTAs, bit for bit,
on both sides of each of the rule's lines."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cloud(n, seed):
    g = torch.Generator().manual_seed(seed)
    v = torch.randn(n - n // 10, 3, generator=g)
    surf = v / v.norm(dim=1, keepdim=True) + 0.005 * torch.randn(n - n // 10, 3, generator=g)
    return torch.cat([surf, 2.4 * torch.rand(n // 10, 3, generator=g) - 1.2]).cuda()


@pytest.mark.parametrize("n,cap,k,kw", [
    (300, 64, 12, {}), (9000, 64, 64, {}), (5000, 100, 16, {}), (65536, 256, 24, {}), (65537, 256, 24, {}),
    (2000, 512, 64, {}), (98304, 512, 16, {}), (98305, 512, 16, {}), (286721, 512, 32, {}),
    (20000, 1000, 32, {}), (393217, 1024, 12, {}), (30000, 2048, 24, {}), (3000, 3000, 12, {}),
    (40000, 512, 16, {"rescore_p2": 1}), (40000, 512, 16, {"stage_off": 3}), (40000, 512, 16, {"stage_off": 4}),
    (40000, 512, 16, {"select_mode": 1, "tau": 8.0}),
])
def test_width_does_not_change_results(n, cap, k, kw):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    xyz = _cloud(n, n + cap)
    d = Denoiser(max_points=n)
    try:
        P = Params(k=k, leaf_capacity=cap, **kw)
        a = d.run(xyz, P)
        d.set_tuning(leaf_threads=128)
        b = d.run(xyz, P)
        assert torch.equal(a.mask, b.mask) and torch.equal(a.stage, b.stage)
        assert torch.equal(a.score.view(torch.int32), b.score.view(torch.int32))
    finally:
        d.close()
