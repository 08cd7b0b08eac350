"""Frames whose views get low and high screen tiles, at CTA sizes with more warps than a low tile has
rows: the pixels of the default size, and the oracle's work list."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shapes", [[(1, 1)], [(130, 9)], [(257, 63), (64, 7)], [(128, 32 * 607)], [(128, 32 * 607 + 1)], [(128, 32 * 1216)],
                                    [(2049, 1150), (2048, 1100)]])
@pytest.mark.parametrize("filt", [0, 1])
def test_tiles(shapes, filt):
    import paper_2510_08166_gb300 as jt
    ts = synth.make_texture_set(31, [(64, 64), (100, 60)], [55, 95], [420, 444])
    o = oracle.texset_from(ts)
    rng = np.random.default_rng(len(shapes) + filt)
    ctx = jt.Context(0, max_cache_blocks=1 << 12)
    ctx.upload_set(ts)
    default = ctx.tuning()
    gbs = []
    for w, h in shapes:
        y, x = np.meshgrid(np.arange(h), np.arange(w), indexing="ij")
        uv = np.stack([x / 701.0 + y / 997.0, y / 503.0 - x / 887.0], -1).astype(np.float32)
        tex = ((x // 37 + y // 23) % 3).astype(np.uint16)
        tex[tex == 2] = 0xFFFF
        mip = rng.integers(0, 2, (h // 16 + 1, w // 16 + 1)).astype(np.uint8).repeat(16, 0).repeat(16, 1)[:h, :w]
        gbs.append(synth.GBuffer(w, h, uv, tex, np.ascontiguousarray(mip)))
    dgbs = [jt.DeviceGBuffer.from_host(g) for g in gbs]
    want = np.unique(np.concatenate([o.compact(o.mark(g, filt)) for g in gbs]))
    first = None
    for threads in (default["pixel_threads"], 64, 512):
        ctx.set_tuning(**{**default, "pixel_threads": threads})
        outs = [torch.full((g.height, g.width, 4), 7, dtype=torch.uint8, device="cuda") for g in gbs]
        ctx.frame(list(zip(dgbs, outs)), filt)
        ctx.stats()
        np.testing.assert_array_equal(ctx.work_list(), want)
        first = first or outs
        for a, b in zip(first, outs):
            assert torch.equal(a, b)
    for g, out in zip(gbs, first):
        if g.npx > 10 ** 6:
            continue
        d = np.abs(out.cpu().numpy().astype(np.int32) - o.colorize(g.uv, g.tex_id, g.mip, filt).astype(np.int32))
        assert d.max() <= (0 if filt == 0 else 1)
    ctx.close()
