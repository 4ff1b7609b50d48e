"""A large leaf of which the voxel gate leaves few, scattered points: results of the
one-CTA path (a call with per-stage outputs), and no slower than the same leaf with every
point searched (a walk over the leaf's rejected points took 30 times as long)."""

import time

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ONE = 0xFFFFFFFF


def _cloud(n, clumps, per):
    g = torch.Generator(device="cuda").manual_seed(n + clumps)
    x = torch.rand(n, 3, generator=g, device="cuda")
    c = torch.rand(clumps, 1, 3, generator=g, device="cuda") + 1e-5 * torch.rand(clumps, per, 3, generator=g, device="cuda")
    x[: clumps * per] = c.reshape(-1, 3)
    return x[torch.randperm(n, generator=g, device="cuda")].contiguous()


@pytest.mark.parametrize("n,clumps,per,k", [(1_000_000, 20, 10, 32), (60_000, 3, 10, 16), (60_000, 40, 9, 64),
                                            (60_000, 1, 12, 32), (5000, 2, 8, 12)])
def test_few_candidates(n, clumps, per, k):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    x = _cloud(n, clumps, per)
    P = Params(k=k, leaf_capacity=ONE, beta=0.5, min_vox_count=8)
    d = Denoiser(max_points=n)
    try:
        r = d.run(x, P)
        n1 = d.stats()["n_p1"]
        assert 0 < n1 <= 2 * clumps * per
        g = d.run_debug(x, P)
        assert torch.equal(r.mask, g["mask"]) and torch.equal(r.stage, g["stage"])
        assert torch.equal(r.score.view(torch.int32), g["score"].view(torch.int32))
        if n < 1_000_000:
            return
        t = {}
        for name, Q in (("few", P), ("all", Params(k=k, leaf_capacity=ONE, min_vox_count=1))):
            o = d.run(x, Q)
            torch.cuda.synchronize()
            a = time.perf_counter()
            for _ in range(3):
                d.run(x, Q, mask=o.mask, score=o.score, stage=o.stage)
            torch.cuda.synchronize()
            t[name] = (time.perf_counter() - a) / 3
        print(t)
        assert t["few"] <= t["all"], t
    finally:
        d.close()
