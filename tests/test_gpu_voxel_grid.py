"""Voxel occupancy by counters addressed by the grid cell and by the hash table (large
grids: small beta, elongated leaves) against a count of equal cells, exactly."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("beta", [0.02, 0.3, 1.0, 3.0, 50.0])
@pytest.mark.parametrize("shape", ["uniform", "line", "plane", "spike"])
@pytest.mark.parametrize("cap", [40, 512, 3000])
def test_occupancy(beta, shape, cap):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    n = 5000
    x = torch.rand(n, 3, generator=torch.Generator().manual_seed(cap)).cuda()
    x *= {"uniform": torch.tensor([1.0, 1, 1]), "line": torch.tensor([1.0, 1e-4, 1e-5]),
          "plane": torch.tensor([1.0, 1, 0]), "spike": torch.tensor([1.0, 1, 1])}[shape].cuda()
    if shape == "spike":
        x[: n // 2] *= 1e-3
    d = Denoiser(max_points=n)
    try:
        g = d.run_debug(x, Params(k=8, leaf_capacity=cap, beta=beta, min_vox_count=2))
    finally:
        d.close()
    _, leaf = torch.unique(g["leaf_start"], return_inverse=True)
    lo = torch.full((int(leaf.max()) + 1, 3), float("inf"), device="cuda").scatter_reduce(
        0, leaf[:, None].expand(-1, 3), x, "amin")
    v = ((x - lo[leaf]) / g["leaf_h"][:, None]).floor().clamp(max=2097151.0).long()
    cell = torch.cat([leaf[:, None], v], 1)
    _, inv, cnt = torch.unique(cell, dim=0, return_inverse=True, return_counts=True)
    assert torch.equal(cnt[inv].int(), g["vox_count"])
    assert torch.equal(g["stage"] == 1, cnt[inv] < 2)
