"""Incomplete Huffman tables with few long codes and streams that meet their unused prefixes: an MCU
is reported as corrupt exactly when the oracle rejects it, and else has the oracle's texels,
with the tables staged in shared memory and not."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

DC, AC = list(range(12)), [0x00, 0x01, 0x02, 0x11, 0x03, 0x21, 0x12, 0x31, 0xF0, 0x04, 0x41, 0x05]
LENGTHS = {"one short, one long": [1, 16], "a few short, one long": [4] * 11 + [12], "long only": [11] * 12}


def tables(lengths, at):
    bits, vals, _ = synth.standard_huffman()
    bits, vals = bits.copy(), vals.copy()
    for t in at:
        bits[t], vals[t] = 0, 0
        for l in lengths:
            bits[t][l - 1] += 1
        vals[t][:len(lengths)] = (AC if t & 1 else DC)[:len(lengths)]
    return bits, vals


@pytest.mark.parametrize("name", LENGTHS)
@pytest.mark.parametrize("at", [(0, 1, 2, 3), (3,)])
@pytest.mark.parametrize("staged", [True, False])
def test_unused_prefixes_are_rejected(name, at, staged):
    import paper_2510_08166_gb300 as jt
    rng = np.random.default_rng(len(name) + len(at))
    bits, vals = tables(LENGTHS[name], at)
    ctx, o = jt.Context(0, 1 << 12), oracle.TexSet()
    # not staged: the MCU shares a CTA with the last of 255 of a texture with tables of its own
    first = synth.encode(synth.texture(7, 17 * 16, 15 * 16), 80, 420)
    px = []
    if not staged:
        ctx.upload(0, 0, first)
        o.add(0, 0, first)
        px = [((x + 0.5) / 17, (y + 0.5) / 15, 0) for y in range(15) for x in range(17)]
    seen = set()
    for t in range(1, 25):
        n = 64
        ones = rng.choice([0.0, 0.02, 0.1, 0.3, 0.5])  # (zeros decode: the shortest code is zeros)
        scan = np.packbits(rng.random(8 * n) < ones)
        enc = synth.encode(synth.texture(1, 16, 16), 80, 420)
        enc.scan, enc.scan_bits, enc.huff_bits, enc.huff_vals = scan, 8 * n, bits, vals
        ctx.upload(t, 0, enc)
        o.add(t, 0, enc)
        try:
            ref = o.decode_mcu(t, 0, 0, 16)
        except ValueError:
            ref = None
        seen.add(ref is None)
        a = np.array(px + [(0.5, 0.5, t)], np.float32)
        gb = synth.GBuffer(len(a), 1, a[None, :, :2].copy(), a[None, :, 2].astype(np.uint16), np.zeros((1, len(a)), np.uint8))
        ctx.mark(jt.DeviceGBuffer.from_host(gb), jt.FILTER_NEAREST)
        ctx.decode()
        st = ctx.stats(check=False)
        assert bool(st["error_bits"] & jt.DEVERR_CORRUPT) == (ref is None), t
        assert st["needed_blocks"] == len(a)
        if ref is not None:
            assert np.array_equal(ctx.tile((0 if staged else 255) + t - 1, 420), ref), t
    assert True in seen
    ctx.close()
