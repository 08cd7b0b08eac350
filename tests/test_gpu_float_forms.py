"""Float chain where its gathers change form: textures of one MCU (a tap pair wraps inside it), odd
MCU counts (a pair with one MCU), runs that end inside a warp's share, MCUs with none, one and
hundreds of pixels, sizes that are not powers of two, one-pixel views, coordinates far outside.

Bars: a value is a sum of at most 4 x 3 x 64 products with every factor below its texels'
scale, so its fp32 error stays below 1e-6 of the frame's norm; a gradient sums up to a few
thousand terms in any order, so its stays below sqrt(n) 2^-24 < 1e-5 of the gradient's norm."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("T,mx,my,W,H,kind", [
    (1, 1, 1, 1, 1, "spread"),       # one pixel, one MCU, both axes wrap inside it
    (3, 1, 1, 65, 17, "spread"),     # an odd number of MCUs, hundreds of pixels in each
    (2, 1, 5, 130, 9, "spread"),     # wrap inside one MCU along x only
    (1, 5, 1, 40, 30, "far"),        # coordinates up to +-3000 (the general taps), not a power of two
    (5, 3, 7, 127, 65, "spread"),    # 105 MCUs: the last warp's share and pair are ragged
    (2, 16, 8, 200, 64, "point"),    # one MCU holds thousands of entries, the others none
    (7, 9, 4, 64, 64, "sparse"),     # few pixels: MCUs with none beside MCUs with one
    (4, 32, 32, 320, 180, "seam"),   # taps on MCU seams and corners: up to four entries per pixel
])
def test_forms(T, mx, my, W, H, kind):
    import paper_2510_08166_gb300 as jt
    rng = np.random.default_rng(T * 1000 + mx * 31 + my)
    coef = (rng.standard_normal((T, my, mx, 6, 64)) * 40).astype(np.float32)
    tex = rng.integers(0, T, (H, W)).astype(np.uint16)
    uv = rng.random((H, W, 2)).astype(np.float32)
    if kind == "far":
        uv = ((uv - 0.5) * 6000).astype(np.float32)
    elif kind == "point":
        uv = (0.5 + uv * 0.01).astype(np.float32)
    elif kind == "sparse":
        tex[rng.random((H, W)) < 0.97] = 0xFFFF
    elif kind == "seam":
        n = np.array([mx, my])
        uv = (np.round(uv * n) / n + rng.choice([0.0, 1e-4], (H, W, 2))).astype(np.float32)
    gb = synth.GBuffer(W, H, uv, tex, np.zeros((H, W), np.uint8))
    ctx = jt.Context(0, 1 << 14)
    ctx.register_coeff_textures(0, T, mx * 16, my * 16)
    dgb = jt.DeviceGBuffer.from_host(gb)
    c = torch.from_numpy(coef).cuda()
    F = torch.empty((H, W, 3), dtype=torch.float32, device="cuda")
    target = rng.random((H, W, 3)).astype(np.float32) * 255
    F_ref = oracle.float_forward(coef, gb)
    _, g_ref = oracle.float_loss_grad(coef, gb, target)
    # the gradient of sum (F - target)^2 from the oracle's own frame: a backward of exact inputs
    gF = torch.from_numpy((2.0 * (F_ref - target)).astype(np.float32)).cuda()
    for _ in range(2):  # the second pass meets what the first one left in the counts
        ctx.colorize_float(dgb, c, F)
        f = F.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(f - F_ref) < 1e-6 * np.linalg.norm(F_ref)
        g = torch.full_like(c, float("nan"))
        ctx.colorize_backward(dgb, gF, g)
        ctx.stats()
        g = g.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(g - g_ref) < 1e-5 * np.linalg.norm(g_ref)
        untouched = np.abs(g_ref).reshape(-1, 384).sum(axis=1) == 0
        assert not g.reshape(-1, 384)[untouched].any()
    ctx.close()
