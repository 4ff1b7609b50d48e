"""Radius counts (Sec. 2.2 baseline) where a sphere's border is settled by boxes of 8
points: clouds that end inside such a box or at its edge, and border lists longer than
the kernel holds (uniform, 119,999 points, R = 0.4 of the extent: half of the warps list
more than 768 chunks).  Whole numbers, equal to a full FP32 comparison."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,radius", [(32_768, 0.2), (32_769, 0.2), (32_775, 0.1), (32_776, 0.3), (32_777, 0.05), (32_799, 0.2),
                                      (119_999, 0.4)])
def test_counts_at_quarter_edges(n, radius):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser
    # R = 6 (sum of the box's face areas) / n: 18 s^2 / n for a cube of side s
    x = (torch.rand(n, 3, generator=torch.Generator().manual_seed(n)) * (radius * n / 18)).cuda()
    d = Denoiser(max_points=n)
    g = d.run_baseline(x, counts=True)
    d.close()
    r2 = g["R"] * g["R"]
    for s in range(0, n, 500):
        d3 = x[None, :, :] - x[s:s + 500, None, :]
        t = d3[..., 0] * d3[..., 0]
        t = (t.double() + d3[..., 1].double() ** 2).float()  # one rounding, as a fused multiply-add
        t = (t.double() + d3[..., 2].double() ** 2).float()
        assert torch.equal((t.double() <= r2).sum(1).int(), g["n_i"][s:s + 500].int())
