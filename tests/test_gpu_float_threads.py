"""The float chain at every CTA size that the tuning accepts: the same gradients."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("threads", [64, 256, 768, 1024])
def test_cta_sizes(threads):
    import paper_2510_08166_gb300 as jt
    gen = torch.Generator("cuda").manual_seed(5)
    w, h = 301, 77
    gb = jt.DeviceGBuffer.empty(w, h)
    gb.uv.copy_(torch.rand((h, w, 2), device="cuda", generator=gen) * 4 - 2)
    gb.tex_id.zero_()
    gb.mip.zero_()
    coef = torch.randn((1, 4, 4, 6, 64), device="cuda", generator=gen)
    grad = torch.randn((h, w, 3), device="cuda", generator=gen)
    got = []
    for t in (256, threads):
        ctx = jt.Context(0, max_cache_blocks=1 << 8)
        ctx.register_coeff_textures(0, 1, 64, 64)
        ctx.set_tuning(**{**ctx.tuning(), "pixel_threads": t})
        c = coef.clone().requires_grad_(True)
        frame = ctx.colorize_float_autograd(gb, c)
        got.append((frame.detach(), torch.autograd.grad(frame, c, grad)[0]))
        ctx.stats()
        ctx.close()
    # the sums differ in their order alone: some hundreds of terms of size 4 at 2^-24 each
    for a, b in zip(*got):
        assert (a - b).abs().max() <= 2e-4
