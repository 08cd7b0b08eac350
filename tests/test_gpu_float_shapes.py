"""Float chain at the sizes where its gathers take other shapes: MCU counts around the steps of pairs
per warp and warps per CTA (ragged ends at each), and MCUs whose pixels are taken in runs.

Bars as for the forms: values within 1e-6 of the frame's norm, gradients within 1e-5 of theirs."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("T,mx,my,W,H,zoom", [
    (1, 1, 1, 200, 37, 0.0),       # thousands of pixels on one MCU
    (1, 3, 101, 130, 50, 0.0),     # one pair a warp, one warp a CTA
    (1, 2, 1, 64, 16, 0.0),        # 1024 pixels on the pair's inner texels and more on its seam: both walks
    (1, 35, 35, 301, 77, 0.03),    # 613 pairs, most pixels in a few MCUs
    (1, 51, 50, 90, 60, 0.0),      # 1275 pairs
    (1, 160, 161, 90, 60, 0.0),    # 12,880: two pairs a warp backwards
    (3, 131, 131, 90, 60, 0.0),    # 25,742: four backwards, two forwards
    (5, 131, 129, 90, 60, 0.01),   # 42,248: eight forwards
])
def test_shapes(T, mx, my, W, H, zoom):
    import paper_2510_08166_gb300 as jt
    rng = np.random.default_rng(T * 1000 + mx * 31 + my)
    coef = (rng.standard_normal((T, my, mx, 6, 64), np.float32) * 40).astype(np.float32)
    uv = rng.random((H, W, 2)).astype(np.float32)
    if zoom:  # pixels in order on a small part, whole runs of them on a texel
        y, x = np.mgrid[0:H, 0:W]
        uv = (0.4 + zoom * np.stack([x / W, y / H], -1)).astype(np.float32)
    # the last MCU, in the last ragged pair, has pixels
    uv[-1, -4:] = 1.0 - 1e-3 / max(mx, my)
    gb = synth.GBuffer(W, H, uv, rng.integers(0, T, (H, W)).astype(np.uint16), np.zeros((H, W), np.uint8))
    gb.tex_id[-1, -4:] = T - 1
    ctx = jt.Context(0, T * mx * my)
    ctx.register_coeff_textures(0, T, mx * 16, my * 16)
    dgb, c = jt.DeviceGBuffer.from_host(gb), torch.from_numpy(coef).cuda()
    F = torch.empty((H, W, 3), dtype=torch.float32, device="cuda")
    F_ref = oracle.float_forward(coef, gb)
    target = rng.random((H, W, 3)).astype(np.float32) * 255
    _, g_ref = oracle.float_loss_grad(coef, gb, target)
    gF = torch.from_numpy((2.0 * (F_ref - target)).astype(np.float32)).cuda()
    for _ in range(2):
        ctx.colorize_float(dgb, c, F)
        assert np.linalg.norm(F.cpu().numpy() - F_ref) < 1e-6 * np.linalg.norm(F_ref)
        g = torch.full_like(c, float("nan"))
        ctx.colorize_backward(dgb, gF, g)
        ctx.stats()
        g = g.cpu().numpy()
        assert np.linalg.norm(g - g_ref) < 1e-5 * np.linalg.norm(g_ref)
        assert not g.reshape(-1, 384)[~g_ref.reshape(-1, 384).any(axis=1)].any()
    ctx.close()
