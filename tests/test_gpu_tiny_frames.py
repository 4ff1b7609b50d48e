"""Batches of small frames under a large leaf capacity: results of each frame's own call,
and a leaf stage as fast as under a capacity of the frames' size.

Tolerance of the time: the capacity may make the stage half as long again."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cloud(n, seed):
    g = torch.Generator().manual_seed(seed)
    v = torch.randn(n, 3, generator=g)
    return (v / v.norm(dim=1, keepdim=True) + 0.01 * torch.randn(n, 3, generator=g)).cuda()


@pytest.mark.parametrize("sizes", [[1, 2, 20, 64, 65, 3], [128, 129, 40, 0, 256], [257, 5, 600], [1500, 30, 700]])
@pytest.mark.parametrize("cap", [16, 64, 512, 2048, 0xFFFFFFFF])
def test_frames_alone_and_together(sizes, cap):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    parts = [_cloud(n, 7 * n + i) for i, n in enumerate(sizes)]
    offs = [0]
    for p in parts:
        offs.append(offs[-1] + len(p))
    d = Denoiser(max_points=offs[-1], max_frames=len(parts))
    try:
        P = Params(k=8, leaf_capacity=cap, min_vox_count=2)
        b = d.run_batch(torch.cat(parts), offs, P)
        for f, p in enumerate(parts):
            if len(p) == 0:
                continue
            r = d.run_debug(p, P)
            for a, c in ((r["mask"], b.mask), (r["stage"], b.stage), (r["score"], b.score)):
                assert torch.equal(a, c[offs[f]:offs[f + 1]])
    finally:
        d.close()


def _stage(frames, m, cap, stage):
    from paper_2512_10386_gb300 import Denoiser, Params
    x = _cloud(frames * m, 3)
    offs = [i * m for i in range(frames + 1)]
    d = Denoiser(max_points=len(x), max_frames=frames)
    try:
        d.set_profiling(True)
        t = []
        for _ in range(12):
            d.run_batch(x, offs, Params(k=8, leaf_capacity=cap))
            t.append(d.stats()["stage_ms"][stage])
        return sorted(t)[6]
    finally:
        d.close()


@pytest.mark.parametrize("m", [20, 100])
def test_leaf_stage_of_small_frames(m):
    import __graft_entry__
    __graft_entry__.build()
    small, large = _stage(3000, m, 64 if m == 20 else 128, 4), _stage(3000, m, 512, 4)
    print(small, large)
    assert large <= 1.5 * small, (small, large)


def test_leaf_finder_of_small_frames():
    import __graft_entry__
    __graft_entry__.build()
    # under a capacity of 8 the finder searches every frame, above 20 there is nothing to search
    search, whole = _stage(3000, 20, 8, 2), _stage(3000, 20, 2048, 2)
    print(search, whole)
    assert whole <= search, (search, whole)


@pytest.mark.parametrize("kw", [{"max_depth": 1}, {"max_depth": 0}, {"leaf_capacity": 0xFFFFFFFF}, {"leaf_capacity": 2000}])
def test_no_launches_for_leaves_that_cannot_be(kw):
    """Whether a batch can hold large leaves is a question of its largest frame: 400 frames
    of 500 points launch what 2 such frames launch."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    n = {}
    for frames in (2, 400):
        x = _cloud(500 * frames, 3)
        d = Denoiser(max_points=len(x), max_frames=frames)
        try:
            d.run_batch(x, [500 * i for i in range(frames + 1)], Params(k=8, **kw))
            n[frames] = d.stats()["launches"]
        finally:
            d.close()
    assert n[400] <= n[2] + 1, n  # (small leaves may take a launch of their own)


@pytest.mark.parametrize("m", [600, 800, 1300])
def test_leaf_stage_of_frames_just_above_the_capacity(m):
    """Frames of which one octree level makes leaves of less than half the capacity: the same
    leaves under a capacity of 256 and 512, so about the same leaf stage (within a quarter)."""
    import __graft_entry__
    __graft_entry__.build()
    g = torch.Generator().manual_seed(9)
    from paper_2512_10386_gb300 import Denoiser, Params
    x = torch.rand(64 * m, 3, generator=g).cuda()
    offs, ms = [i * m for i in range(65)], {}
    d = Denoiser(max_points=len(x), max_frames=64)
    try:
        d.set_profiling(True)
        masks = {}
        for cap in (256, 512):
            t = []
            for _ in range(12):
                masks[cap] = d.run_batch(x, offs, Params(k=12, leaf_capacity=cap)).mask
                t.append(d.stats()["stage_ms"][4])
            ms[cap] = sorted(t)[6]
    finally:
        d.close()
    print(ms)
    assert torch.equal(masks[256], masks[512])
    assert ms[512] <= 1.25 * ms[256], ms
