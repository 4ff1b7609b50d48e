"""The pruned cross-set passes (large pairs of clouds) against full comparisons:
nearest squared distances against the full pass's (which a small query cloud
takes), counts within the radius against a chunked FP32 comparison, bit for bit."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def den():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser
    d = Denoiser(max_points=120_000)
    yield d
    d.close()


def _cloud(kind, n, seed):
    g = torch.Generator().manual_seed(seed)
    r = torch.rand(n, 3, generator=g)
    if kind == "surface":
        v = torch.randn(n, 3, generator=g)
        x = v / v.norm(dim=1, keepdim=True) + 0.003 * torch.randn(n, 3, generator=g)
        x[: n // 10] = 3 * r[: n // 10] - 1.5
        return x[torch.randperm(n, generator=g)]
    if kind == "clusters":
        return r[torch.randint(37, (n,), generator=g)] + 1e-4 * torch.randn(n, 3, generator=g)
    if kind == "duplicates":
        return r[torch.randint(50, (n,), generator=g)].clone()
    if kind == "line":
        return r * torch.tensor([1.0, 0.0, 0.0])
    if kind == "huge":
        return (r - 0.5) * 3e38
    return r  # uniform


@pytest.mark.parametrize("kind,na,nb", [("surface", 50_000, 51_237), ("uniform", 32_768, 16_384), ("clusters", 33_001, 19_999),
                                        ("duplicates", 25_000, 22_011), ("line", 22_385, 30_000), ("huge", 24_000, 24_001),
                                        ("surface", 100_000, 5_370), ("uniform", 5_400, 99_999)])
def test_nearest_equals_the_full_pass(den, kind, na, nb):
    a, b = _cloud(kind, na, 1).cuda(), _cloud(kind, nb, 2).cuda()
    g = den.eval_metrics(a, b, per_point=True)
    for q, c, got in ((a, b, g["nn_clean"]), (b, a, g["nn_denoised"])):
        step = (1 << 29) // len(c) - 1  # below the line: every pair is compared
        for s in range(0, len(q), max(step, len(q) // 3)):
            e = min(len(q), s + step)
            part = den.eval_metrics(q[s:e].contiguous(), c, per_point=True)["nn_clean"]
            assert torch.equal(part.view(torch.int32), got[s:e].view(torch.int32))


@pytest.mark.parametrize("kind,n,scale", [("surface", 40_000, 1.0), ("surface", 40_000, 30.0), ("surface", 40_001, 400.0),
                                          ("surface", 32_768, 1e5), ("uniform", 33_333, 200.0), ("clusters", 34_000, 60.0),
                                          ("duplicates", 37_000, 30.0), ("line", 36_385, 1.0)])
def test_counts_equal_the_full_comparison(den, kind, n, scale):
    x = (_cloud(kind, n, 3) * scale).cuda()
    g = den.run_baseline(x, counts=True)
    r2 = torch.tensor(g["R"] * g["R"], dtype=torch.float64)
    for s in range(0, n, 2000):
        d = x[None, :, :] - x[s:s + 2000, None, :]
        t = (d[..., 0] * d[..., 0]).double()
        t = (t + d[..., 1].double() ** 2).float().double()
        d2 = (t + d[..., 2].double() ** 2).float()
        want = (d2.double() <= r2.item()).sum(1)
        assert torch.equal(want.int(), g["n_i"][s:s + 2000])
