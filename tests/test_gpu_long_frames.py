"""Frames of many tiles: the keys of a frame whose extremes lie in its first and last
tiles, alone and between short frames, and the time of the front end's first passes,
which must grow with the points and not with their square.

Tolerance of the time: 16 times the points may take 32 times as long."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _keys(x):
    lo = x.amin(0)
    s = torch.tensor(2097152.0, device="cuda") / (x.amax(0) - lo).amax()
    q = ((x - lo) * s).floor().clamp(max=2097151.0).long()
    key = torch.zeros(len(x), dtype=torch.int64, device="cuda")
    for b in range(21):
        for a in range(3):
            key |= ((q[:, a] >> b) & 1) << (3 * b + 2 - a)
    return key


def _cloud(n, seed):
    x = torch.rand(n, 3, generator=torch.Generator(device="cuda").manual_seed(seed), device="cuda")
    x[0] = -1.0
    x[-1] = torch.tensor([2.0, 1.5, 1.25], device="cuda")
    return x


@pytest.mark.parametrize("tiles", [1023, 1024, 1025, 2500])
def test_keys_and_batches(tiles):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    n, P = 2048 * tiles - 700, Params(k=4, leaf_capacity=64)
    x = _cloud(n, tiles)
    parts = [_cloud(3000, 1), x, _cloud(5, 2), x[: n // 2].contiguous(), _cloud(9000, 3)]
    offs = [0]
    for p in parts:
        offs.append(offs[-1] + len(p))
    d = Denoiser(max_points=offs[-1], max_frames=len(parts))
    try:
        g = d.run_debug(x, P)
        assert torch.equal(g["key"], _keys(x))
        b = d.run_batch(torch.cat(parts), offs, P)
        for f, p in enumerate(parts):
            r = d.run(p, P)
            assert torch.equal(r.mask, b.mask[offs[f]:offs[f + 1]])
            assert torch.equal(r.score, b.score[offs[f]:offs[f + 1]])
        x[n // 2] = float("nan")
        with pytest.raises(Exception, match="NaN"):
            d.run(x, P)
    finally:
        d.close()


def test_first_passes_grow_with_the_points():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser, Params
    big = 64 << 20
    x = _cloud(big, 7)
    d = Denoiser(max_points=big)
    ms = []
    try:
        d.set_profiling(True)
        for n in (big // 16, big):
            t = []
            for _ in range(6):
                d.run(x[:n], Params(k=4, leaf_capacity=64))
                t.append(d.stats()["stage_ms"][0])
            ms.append(sorted(t)[2])
    finally:
        d.close()
    assert ms[1] <= 32.0 * ms[0], ms
