"""Small clouds with one point far away: the others share one node of the sorted depth,
whose order the one-block front end completes.  Results of the general path (a call with
a look-back hook on a tile that does not exist), leaves against the oracle's, and a time
that does not grow with the node's size times the capacity.

Tolerance of the time: the far point may make the call twice as long."""

import time

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cloud(n, far):
    g = torch.Generator().manual_seed(n)
    v = torch.randn(n - n // 10, 3, generator=g)
    surf = v / v.norm(dim=1, keepdim=True) + 0.005 * torch.randn(n - n // 10, 3, generator=g)
    x = torch.cat([surf, 2.4 * torch.rand(n // 10, 3, generator=g) - 1.2])[torch.randperm(n, generator=g)]
    if far:
        x[n // 2] = far
    return x.cuda().contiguous()


@pytest.mark.parametrize("n", [2, 700, 1500, 4096])
@pytest.mark.parametrize("cap", [1, 64, 512, 1024, 2048, 4095])
@pytest.mark.parametrize("far", [30.0, 3e3, 3e4, 1e7])
def test_against_the_general_path(n, cap, far):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    x = _cloud(n, far)
    d = Denoiser(max_points=n)
    try:
        P = Params(k=8, leaf_capacity=cap, min_vox_count=1)
        a = d.run_debug(x, P)
        d.test_hold_lookback(1 << 20)
        b = d.run_debug(x, P)
        for name in ("key", "leaf_start", "leaf_count", "leaf_h", "mask", "stage", "score", "nbr"):
            assert torch.equal(a[name], b[name]), name
    finally:
        d.close()


def test_time_with_a_far_point():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    ms = {}
    d = Denoiser(max_points=4096)
    try:
        d.set_profiling(True)
        for far in (None, 3e4):
            x, t = _cloud(4096, far), []
            for _ in range(12):
                d.run(x, Params(k=12, leaf_capacity=1024))
                t.append(d.stats()["stage_ms"][0])  # the one-block front end
            ms[far] = sorted(t)[6]
    finally:
        d.close()
    print(ms)
    assert ms[3e4] <= 2.0 * ms[None], ms
