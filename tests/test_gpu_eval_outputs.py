"""Metrics whose two distance outputs are one buffer, or overlap: the metrics of a call
without outputs, and the denoised cloud's distances in the shared part (they come last)."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("na,nb", [(2000, 2000), (33_000, 33_000), (40_000, 30_000)])
@pytest.mark.parametrize("shift", [0, 500])
def test_overlapping_outputs(na, nb, shift):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser
    from paper_2512_10386_gb300 import _native as N
    g = torch.Generator(device="cuda").manual_seed(na)
    a = torch.rand(na, 3, generator=g, device="cuda")
    b = torch.rand(nb, 3, generator=g, device="cuda") + 0.01
    d = Denoiser(max_points=max(na, nb))
    try:
        want = d.eval_metrics(a, b, per_point=True)
        out = torch.zeros(max(na, nb) + 500, device="cuda")
        torch.cuda.synchronize()
        st, m = N.denoise_eval_metrics(d.ctx, a.data_ptr(), na, b.data_ptr(), nb, out.data_ptr(),
                                       out[shift:].data_ptr(), None)
        assert st == 0
        assert (m[0], m[1], m[2]) == (want["mse"], want["chamfer"], want["psnr"])
        assert torch.equal(out[shift:shift + nb], want["nn_denoised"])
        assert torch.equal(out[:shift], want["nn_clean"][:shift])
    finally:
        d.close()


@pytest.mark.parametrize("n", [2000, 33_000])
@pytest.mark.parametrize("off_a,off_b", [(1, 0), (0, 2), (3, 3)])
def test_outputs_at_any_byte(n, off_a, off_b):
    """Distance buffers that are not aligned for floats: copied to, never stored to."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_10386_gb300 import Denoiser
    from paper_2512_10386_gb300 import _native as N
    g = torch.Generator(device="cuda").manual_seed(n)
    a = torch.rand(n, 3, generator=g, device="cuda")
    b = torch.rand(n, 3, generator=g, device="cuda") + 0.01
    d = Denoiser(max_points=n)
    try:
        want = d.eval_metrics(a, b, per_point=True)
        x, y = (torch.zeros(4 * n + 8, dtype=torch.uint8, device="cuda") for _ in range(2))
        torch.cuda.synchronize()
        st, m = N.denoise_eval_metrics(d.ctx, a.data_ptr(), n, b.data_ptr(), n, x.data_ptr() + off_a,
                                       y.data_ptr() + off_b, None)
        assert st == 0
        assert (m[0], m[1], m[2]) == (want["mse"], want["chamfer"], want["psnr"])
        assert torch.equal(x[off_a:off_a + 4 * n], want["nn_clean"].view(torch.uint8))
        assert torch.equal(y[off_b:off_b + 4 * n], want["nn_denoised"].view(torch.uint8))
    finally:
        d.close()
