"""Values that are not finite in the float chain go where their weights are not zero: a texel of weight
zero, as pixels on texel centres have three of, changes neither the value nor the gradient."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

W = H = 64  # one pixel per texel of a 4 x 4 MCU texture, on its centre


def setup():
    import paper_2510_08166_gb300 as jt
    y, x = np.mgrid[0:H, 0:W]
    uv = np.stack([(x + 0.5) / W, (y + 0.5) / H], -1).astype(np.float32)
    gb = synth.GBuffer(W, H, uv, np.zeros((H, W), np.uint16), np.zeros((H, W), np.uint8))
    ctx = jt.Context(0, 64)
    ctx.register_coeff_textures(0, 1, W, H)
    return ctx, jt.DeviceGBuffer.from_host(gb)


@pytest.mark.parametrize("bad", [float("inf"), float("-inf"), float("nan")])
@pytest.mark.parametrize("du", [0, 3, 4, 5])
def test_a_coefficient(bad, du):
    ctx, gb = setup()
    coef = torch.randn((1, 4, 4, 6, 64), generator=torch.Generator().manual_seed(3)) * 20
    out = torch.empty((H, W, 3), device="cuda")
    ctx.colorize_float(gb, coef.cuda(), out)
    want = out.cpu()
    coef[0, 2, 1, du, 0] = bad  # the DC of one data unit: every texel of it
    ctx.colorize_float(gb, coef.cuda(), out)
    got = out.cpu()
    y, x = torch.meshgrid(torch.arange(H), torch.arange(W), indexing="ij")
    y0, x0, n = {0: (32, 16, 8), 3: (40, 24, 8)}.get(du, (32, 16, 16))
    hit = (y >= y0) & (y < y0 + n) & (x >= x0) & (x < x0 + n)
    assert torch.equal(got[~hit], want[~hit])
    # luma is in all three channels, Cb not in red, Cr not in blue
    for c, sign in enumerate({4: (0, -1, 1), 5: (1, -1, 0)}.get(du, (1, 1, 1))):
        g = got[hit][:, c]
        if sign == 0:
            assert torch.equal(g, want[hit][:, c])
        elif bad != bad:
            assert g.isnan().all()
        else:
            assert (g == sign * bad).all()
    ctx.close()


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_a_pixel_s_gradient(bad):
    ctx, gb = setup()
    grad = torch.randn((H, W, 3), generator=torch.Generator().manual_seed(4)).cuda()
    out = torch.empty((1, 4, 4, 6, 64), device="cuda")
    ctx.colorize_backward(gb, grad, out)
    want = out.clone()
    grad[31, 15, 1] = bad  # the last texel of MCU (1, 0), next to three others
    ctx.colorize_backward(gb, grad, out)
    spoilt = torch.zeros(out.shape, dtype=torch.bool, device="cuda")
    spoilt[0, 1, 0, [3, 4, 5]] = True  # its data unit and its chroma
    assert not out[spoilt].isfinite().any()
    # (the others' sums differ in their order alone: four terms of size 8 at 2^-24 each)
    assert (out - want)[~spoilt].abs().max() <= 1e-5
    ctx.close()
