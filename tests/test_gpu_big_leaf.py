"""Leaves spread over the whole GPU against the one-CTA path (which a call with
per-stage outputs takes): masks, stages and scores bit for bit, over the leaf
sizes, orders and degenerate clouds where the two could part."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ONE = 0xFFFFFFFF


def _surface(n, seed):
    g = torch.Generator().manual_seed(seed)
    v = torch.randn(n - n // 10, 3, generator=g)
    surf = v / v.norm(dim=1, keepdim=True) + 0.005 * torch.randn(n - n // 10, 3, generator=g)
    return torch.cat([surf, 2.4 * torch.rand(n // 10, 3, generator=g) - 1.2])


def _lattice(m, step):
    a = torch.arange(m, dtype=torch.float32) * step
    x = torch.stack(torch.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3)
    return x[torch.randperm(len(x), generator=torch.Generator().manual_seed(m))]


def _dups(n, kinds):
    g = torch.Generator().manual_seed(n)
    return torch.rand(kinds, 3, generator=g)[torch.randint(kinds, (n,), generator=g)]


def _check(xyz, offsets=None, **kw):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    xyz = xyz.cuda().contiguous()
    offsets = offsets or [0, len(xyz)]
    d = Denoiser(max_points=len(xyz), max_frames=len(offsets) - 1)
    try:
        P = Params(**kw)
        a = d.run_batch(xyz, offsets, P)
        s = d.stats()
        tot = {k: 0 for k in ("knn_pairs", "n_p1", "n_p2", "score_terms")}
        for f in range(len(offsets) - 1):
            b, e = offsets[f], offsets[f + 1]
            r = d.run_debug(xyz[b:e].contiguous(), P)
            assert torch.equal(a.mask[b:e], r["mask"]) and torch.equal(a.stage[b:e], r["stage"])
            assert torch.equal(a.score[b:e].view(torch.int32), r["score"].view(torch.int32))
            for k in tot:
                tot[k] += d.stats()[k]
        assert {k: s[k] for k in tot} == tot
    finally:
        d.close()


@pytest.mark.parametrize("n", [513, 545, 1023, 1024, 1025, 2049, 4097])
@pytest.mark.parametrize("k", [1, 12, 32, 64])
def test_one_leaf_sizes(n, k):
    _check(_surface(n, n + k), k=k, leaf_capacity=ONE)


@pytest.mark.parametrize("kw", [
    {"max_depth": 0}, {"max_depth": 1, "leaf_capacity": 64}, {"max_depth": 2, "leaf_capacity": 1500},
    {"leaf_capacity": 1025}, {"select_mode": 1, "tau": 8.0}, {"lam": 0.3, "rho_percentile": 40.0},
    {"rho_percentile": 100.0}, {"rho_percentile": 0.0, "gamma": 3.0, "alpha": -0.5, "sigma": 0.7},
    {"min_vox_count": 60}, {"min_vox_count": 4000}, {"k": 33}, {"k": 64},
])
def test_parameters(kw):
    _check(_surface(10000, 5), **{"k": 16, "leaf_capacity": ONE, **kw})


@pytest.mark.parametrize("make", [lambda: _lattice(13, 0.125), lambda: _dups(3000, 7), lambda: _dups(2000, 1),
                                  lambda: _dups(2500, 900), lambda: _surface(3000, 2) * torch.tensor([1., 1., 0.]),
                                  lambda: _surface(3000, 3) * 1e30, lambda: _surface(3000, 4) * 1e-30])
def test_ties_duplicates_and_scales(make):
    _check(make(), k=12, leaf_capacity=ONE, min_vox_count=2)
    _check(make(), k=32, leaf_capacity=1100, max_depth=4, min_vox_count=1)


def test_batch_of_one_leaf_frames_and_small_leaves():
    parts = [_surface(n, n) for n in (1, 700, 40, 2100, 5, 1500)]
    offs = [0]
    for p in parts:
        offs.append(offs[-1] + len(p))
    _check(torch.cat(parts), offs, k=8, leaf_capacity=ONE)
    _check(torch.cat(parts), offs, k=8, leaf_capacity=1100)


@pytest.mark.parametrize("n,cap,k,kw", [
    (3000, 512, 12, {}), (20_000, 256, 32, {}), (20_000, 64, 1, {}), (5000, ONE, 24, {}), (9000, 30, 20, {}),
    (9000, 128, 32, {"max_depth": 2}), (4000, 512, 16, {"min_vox_count": 40}), (1, 512, 8, {}), (33, 8, 32, {}),
])
@pytest.mark.parametrize("make", ["surface", "lattice", "dups"])
def test_cross_leaf_box_search_against_the_lists(n, cap, k, kw, make):
    """Cross-leaf neighbours of the box search (K <= 32) against the exhaustive lists, which
    K = 33 takes: the first K of the 33 in (d^2, input index) order are the K nearest."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    if make == "surface":
        xyz = _surface(n, n + k)
    elif make == "lattice":
        xyz = _lattice(max(2, round(n ** (1 / 3))), 0.125)
    else:
        xyz = _dups(n, max(1, n // 9))
    xyz = xyz.cuda().contiguous()
    d = Denoiser(max_points=len(xyz))
    try:
        d.set_cross_leaf(True)
        kw = {"leaf_capacity": cap, "cross_leaf": 1, "min_vox_count": 2, **kw}
        a = d.run_debug(xyz, Params(k=k, **kw))
        b = d.run_debug(xyz, Params(k=33, **kw))
        p1 = b["stage"] != 1
        assert torch.equal(a["nbr"][p1], b["nbr"][p1][:, :k])
        assert torch.equal(a["nbr_d2"][p1], b["nbr_d2"][p1][:, :k])
        r = d.run(xyz, Params(k=k, **kw))
        assert torch.equal(r.mask, a["mask"]) and torch.equal(r.score, a["score"])
    finally:
        d.close()
