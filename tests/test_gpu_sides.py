"""Colourise's repeat wrap against the oracle for levels of every kind of side: one texel, odd
sides, powers of two beside others; coordinates on texel and repeat edges, negative, far out, and
beyond the fast path's range."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIDES = [(1, 1), (3, 1), (1, 7), (17, 33), (100, 64), (255, 257), (549, 5), (16, 16), (9, 2047)]


def _uv(rng, w, h, n):
    """Coordinates in texels of a w x h level, as uv."""
    parts = []
    for side in (w, h):
        k = rng.integers(-3 * side - 2, 3 * side + 3, n).astype(np.float64)
        k += rng.choice([0, 0.5, -2.0 ** -8, 2.0 ** -8, 0.25], n)
        far = rng.random(n)
        k = np.where(far < 0.15, k + side * np.floor(2.0 ** 21 / side * rng.uniform(-1, 1, n)), k)
        k = np.where((far >= 0.15) & (far < 0.2), k + rng.choice([-1, 1], n) * 2.0 ** rng.integers(22, 30, n), k)
        parts.append((k / side).astype(np.float32))
    return np.stack(parts, -1)


@pytest.mark.parametrize("filt", [0, 1, 2])
@pytest.mark.parametrize("plain", [False, True])
def test_wrap(filt, plain):
    import paper_2510_08166_gb300 as jt
    rng = np.random.default_rng(7 + filt)
    ts = synth.TextureSet([[synth.encode(synth.texture(synth.mix_seed(5, w, h), w, h), 80, 444 if i % 2 else 420)]
                           for i, (w, h) in enumerate(SIDES)])
    n = 517
    gb = synth.GBuffer(n, len(SIDES), np.stack([_uv(rng, w, h, n) for w, h in SIDES]),
                       np.repeat(np.arange(len(SIDES), dtype=np.uint16)[:, None], n, 1),
                       np.zeros((len(SIDES), n), np.uint8))
    o = oracle.texset_from(ts)
    ctx = jt.Context(0, max_cache_blocks=1 << 12)
    ctx.upload_set(ts)
    dgb = jt.DeviceGBuffer.from_host(gb)
    out = torch.zeros((gb.height, gb.width, 4), dtype=torch.uint8, device="cuda")
    if plain:
        ctx.frame_plain([(dgb, out)], filt)
    else:
        ctx.frame([(dgb, out)], filt)
        np.testing.assert_array_equal(ctx.work_list(), o.compact(o.mark(gb, filt)))
    d = np.abs(out.cpu().numpy().astype(np.int32) - o.colorize(gb.uv, gb.tex_id, gb.mip, filt).astype(np.int32))
    assert d.max() <= (0 if filt == 0 else 1)
    ctx.close()
