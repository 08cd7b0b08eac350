"""Decode of long work lists against the oracle: batches of 32 MCUs in two parts (4:2:0, and both
samplings in one batch), packed (4:4:4), their ragged end, MCUs longer than their share of the
stage, at the narrowest launch shapes, whose lists count as long from a few thousand MCUs."""

import numpy as np
import pytest

import oracle
import synth
from helpers import GidMap, check_tiles, mcu_grid_gbuffer

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("width,warps", [(4, 1), (8, 1), (16, 1), (32, 1), (4, 2)])
@pytest.mark.parametrize("sampling,quality", [((444, 444), 60), ((444, 444), 100), ((420, 420), 75), ((444, 420), 95)])
def test_every_mcu(width, warps, sampling, quality):
    import paper_2510_08166_gb300 as jt
    ctx = jt.Context(0, max_cache_blocks=1 << 18)
    ctx.set_tuning(**{**ctx.tuning(), "decode_mcus_per_warp": width, "decode_warps": warps, "decode_ctas_per_sm": 1})
    need = 11 * torch.cuda.get_device_properties(0).multi_processor_count * width * warps
    # small textures of the two samplings in turn, so that many batches hold both
    w, h = 264, 200
    enc = [synth.encode(synth.texture(9 + i, w, h), quality, s) for i, s in enumerate(sampling)]
    levels, have = [], 0
    while have < need:
        levels.append([enc[len(levels) % 2]])
        have += levels[-1][0].nmcu
    ts = synth.TextureSet(levels)
    ctx.upload_set(ts)
    gb = mcu_grid_gbuffer(ts)
    ctx.mark(jt.DeviceGBuffer.from_host(gb), jt.FILTER_NEAREST)
    ctx.decode()
    ctx.stats()
    work = ctx.work_list()
    assert work.size == have
    o, gm = oracle.texset_from(ts), GidMap(ts)
    # every tile: the textures of one encoding are equal
    slots = ctx.slots(0, have)
    cells = ctx.cache_units(0, int(slots.max()) + 4)
    first, base = {}, 0
    for t, (e,) in enumerate(levels):
        at = slots[base:base + e.nmcu]
        tiles = np.stack([cells[at + u] for u in range(4 if e.sampling == 420 else 1)], 1)
        np.testing.assert_array_equal(tiles, first.setdefault(t % 2, tiles))
        base += e.nmcu
    check_tiles(ctx, o, gm, range(enc[0].nmcu + enc[1].nmcu))
    ctx.close()
