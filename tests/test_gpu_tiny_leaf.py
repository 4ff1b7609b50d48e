"""Leaves of at most 64 points, one warp each, against the fused kernel (which
explicit 64-thread CTAs take): masks, stages, scores and statistics bit for bit, on
surfaces, lattices and duplicates, for every list size and selection rule."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cloud(kind, n):
    g = torch.Generator().manual_seed(n)
    if kind == "surface":
        v = torch.randn(n - n // 10, 3, generator=g)
        surf = v / v.norm(dim=1, keepdim=True) + 0.005 * torch.randn(n - n // 10, 3, generator=g)
        return torch.cat([surf, 2.4 * torch.rand(n // 10, 3, generator=g) - 1.2])
    if kind == "lattice":
        m = round(n ** (1 / 3))
        a = torch.arange(m, dtype=torch.float32) * 0.125
        x = torch.stack(torch.meshgrid(a, a, a, indexing="ij"), -1).reshape(-1, 3)
        return x[torch.randperm(len(x), generator=g)]
    if kind == "duplicates":
        return torch.rand(n // 5, 3, generator=g)[torch.randint(n // 5, (n,), generator=g)]
    return (torch.rand(n, 3, generator=g) - 0.5) * 1e30  # huge


@pytest.mark.parametrize("kind", ["surface", "lattice", "duplicates", "huge"])
@pytest.mark.parametrize("kw", [
    {"k": 1}, {"k": 12}, {"k": 24}, {"k": 31}, {"k": 32}, {"k": 63}, {"k": 64}, {"k": 16, "select_mode": 1, "tau": 6.0},
    {"k": 12, "lam": 0.3, "rho_percentile": 40.0}, {"k": 12, "rho_percentile": 100.0, "lam": 0.01},
    {"k": 9, "gamma": 3.0, "alpha": -0.5, "sigma": 0.7, "eps_k": 1e-3}, {"k": 12, "min_vox_count": 1},
    {"k": 12, "min_vox_count": 9}, {"k": 8, "beta": 0.7, "min_vox_count": 2},
])
def test_tiny_leaves_equal_the_fused_kernel(kind, kw):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    for n, cap in ((81_000, 64), (251_000, 100), (80_001, 33)):
        xyz = _cloud(kind, n).cuda().contiguous()
        d = Denoiser(max_points=len(xyz))
        try:
            P = Params(**{"min_vox_count": 2, "leaf_capacity": cap, **kw})
            a, sa = d.run(xyz, P), d.stats()
            d.set_tuning(leaf_threads=64)
            b, sb = d.run(xyz, P), d.stats()
            assert torch.equal(a.mask, b.mask) and torch.equal(a.stage, b.stage)
            assert torch.equal(a.score.view(torch.int32), b.score.view(torch.int32))
            for k in ("knn_pairs", "n_p1", "n_p2", "score_terms"):
                assert sa[k] == sb[k]
        finally:
            d.close()
