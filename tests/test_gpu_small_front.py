"""The one-block front end of small calls against the tiled one (which a batch of two
frames takes): identical results, over tile and sort edges, deep clusters, depth
limits, host input and rejected input."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def den():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser
    d = Denoiser(max_points=20_000, max_frames=2)
    yield d
    d.close()


def _cloud(kind, n):
    g = torch.Generator().manual_seed(n)
    r = torch.rand(n, 3, generator=g)
    if kind == "surface":
        v = torch.randn(n, 3, generator=g)
        x = v / v.norm(dim=1, keepdim=True)
        x[: n // 10] = 2.4 * r[: n // 10] - 1.2
        return x[torch.randperm(n, generator=g)].contiguous()
    if kind == "clusters":  # cells far below the sorted depth, some points equal
        c = torch.rand(3, 3, generator=g)[torch.randint(3, (n,), generator=g)]
        x = torch.where((torch.arange(n) % 3 == 0)[:, None], r, c + 1e-5 * r)
        x[1::7] = x[0]
        return x.contiguous()
    return r[torch.randint(max(1, n // 4), (n,), generator=g)].contiguous()  # duplicates


def _same(d, xyz, P):
    a = d.run(xyz, P)
    two = torch.cat([xyz, torch.rand(50, 3, device="cuda")]).contiguous()
    b = d.run_batch(two, [0, len(xyz), len(two)], P)
    n = len(xyz)
    assert torch.equal(a.mask, b.mask[:n]) and torch.equal(a.stage, b.stage[:n])
    assert torch.equal(a.score.view(torch.int32), b.score[:n].view(torch.int32))
    return a


@pytest.mark.parametrize("kind", ["surface", "clusters", "duplicates"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 1000, 1024, 1025, 2048, 2049, 3333, 4095, 4096, 4097])
def test_sizes(den, kind, n):
    from paper_2512_10386_gb300 import Params
    xyz = _cloud(kind, n).cuda()
    for cap in (8, 100, 512):
        _same(den, xyz, Params(k=12, leaf_capacity=cap, min_vox_count=2))


@pytest.mark.parametrize("depth", [0, 1, 4, 5, 10, 11, 15, 20])
def test_depth_limits(den, depth):
    from paper_2512_10386_gb300 import Params
    for kind in ("surface", "clusters"):
        _same(den, _cloud(kind, 3000).cuda(), Params(k=8, leaf_capacity=40, max_depth=depth, min_vox_count=1))


def test_host_input_keys_and_rejection(den):
    from paper_2512_10386_gb300 import Params, _native as N
    P = Params(k=12, leaf_capacity=64, min_vox_count=2)
    x = _cloud("clusters", 3100)
    a = _same(den, x.cuda(), P)
    for h in (x.clone(), x.pin_memory()):
        r = den.run(h, P)
        assert torch.equal(r.mask, a.mask.cpu()) and torch.equal(r.score, a.score.cpu())
    bad = x.clone().cuda()
    bad[1234, 1] = float("inf")
    with pytest.raises(N.DenoiseError) as e:
        den.run(bad, P)
    assert e.value.status == N.DENOISE_E_NONFINITE
    _same(den, x.cuda(), P)
