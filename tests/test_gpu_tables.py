"""GPU parity of the decoder's table and staging paths: Huffman tables of every shape (typical,
incomplete, only short codes, only long codes, long codes beyond the second-level entries,
several sets in one context), MCUs longer than the stage, and coefficients at the bounds of
the transform's two column passes. Tiles bit-exact against the oracle."""

import math

import numpy as np
import pytest

import oracle
import synth
from helpers import GidMap, check_tiles, frame, mcu_grid_gbuffer

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

AC_SYMBOLS = [(r << 4) | s for r in range(16) for s in range(1, 11)] + [0x00, 0xF0]


@pytest.fixture(scope="module")
def jt():
    import paper_2510_08166_gb300 as m
    return m


def spec(symbols, length):
    """(bits[16], vals[256]) of canonical codes with length(rank) bits, ranks in symbol order."""
    order = sorted(range(len(symbols)), key=lambda i: (length(i), i))
    bits, vals = np.zeros(16, np.uint8), np.zeros(256, np.uint8)
    for n, i in enumerate(order):
        bits[length(i) - 1] += 1
        vals[n] = symbols[i]
    return bits, vals


def tables(kind):
    if kind == "typical":
        bits, vals, _ = synth.standard_huffman()
        return bits, vals
    ac = {"incomplete": lambda i: min(14, 3 + int(math.log2(1 + i) * 1.6)),  # prefixes left above the last code
          "short": lambda i: 8,       # no code needs a second-level entry
          "long": lambda i: 13,       # every code does, from prefix 0 on
          "walk": lambda i: 11}[kind]  # they take more prefixes than the second level holds
    specs = [spec(range(12), lambda i: 4), spec(AC_SYMBOLS, ac)] * 2
    return np.stack([s[0] for s in specs]), np.stack([s[1] for s in specs])


def encode(coefs, sampling, mx, my, qt, bits, vals):
    """Entropy-codes quantised blocks [nmcu, ndu, 64] (zig-zag order) with the given tables."""
    codes = [synth.encoder_codes(bits[t], vals[t]) for t in range(4)]
    nmcu, ndu, _ = coefs.shape
    out, index, pred = [], np.zeros(nmcu, synth.INDEX_DTYPE), [0, 0, 0]
    total = 0

    def put(t, sym, v, s):
        nonlocal total
        code, length = int(codes[t][0][sym]), int(codes[t][1][sym])
        assert length
        out.append(format(code, f"0{length}b"))
        if s:
            out.append(format(v if v > 0 else v + (1 << s) - 1, f"0{s}b"))
        total += length + s

    for m in range(nmcu):
        index[m]["bit_offset"], index[m]["dc_pred"] = total, pred
        for d in range(ndu):
            comp = 0 if d < ndu - 2 else d - ndu + 3
            cls = 2 if comp else 0
            z = [int(v) for v in coefs[m, d]]
            diff, pred[comp] = z[0] - pred[comp], z[0]
            put(cls, abs(diff).bit_length(), diff, abs(diff).bit_length())
            run = 0
            for k in range(1, 64):
                if z[k] == 0:
                    run += 1
                    continue
                while run > 15:
                    put(cls + 1, 0xF0, 0, 0)
                    run -= 16
                s = abs(z[k]).bit_length()
                put(cls + 1, (run << 4) | s, z[k], s)
                run = 0
            if run:
                put(cls + 1, 0, 0, 0)
    text = "".join(out)
    text += "1" * (-len(text) % 8)
    scan = np.frombuffer(int(text, 2).to_bytes(len(text) // 8, "big"), np.uint8).copy()
    side = 16 if sampling == 420 else 8
    return synth.Encoded(mx * side, my * side, sampling, mx, my, 0, np.zeros(0, np.uint8), scan, total, index, qt, bits, vals)


def blocks(rng, nmcu, ndu, density, amplitude):
    c = np.zeros((nmcu, ndu, 64), np.int64)
    on = rng.random(c.shape) < density
    c[on] = rng.integers(-amplitude, amplitude + 1, int(on.sum()))
    c[:, :, 0] = rng.integers(-1000, 1001, c.shape[:2])
    c[0, 0, 1:] = 0  # DC only
    c[0, 1, 63] = 1  # a run to the last slot
    return c


@pytest.mark.parametrize("kinds", [["typical"], ["incomplete"], ["short"], ["long"], ["walk"],
                                   ["typical", "incomplete", "long", "walk", "short"]])
@pytest.mark.parametrize("density,amplitude,step", [(0.08, 3, 7), (0.9, 900, 1), (0.5, 1023, 255), (0.3, 60, 9)])
@pytest.mark.parametrize("mcus", [4, 16])
def test_tables_and_stages(jt, kinds, density, amplitude, step, mcus):
    rng = np.random.default_rng(len(kinds) * 1000 + amplitude + mcus)
    levels = []
    for n, kind in enumerate(kinds):
        sampling, mx, my = (420, 5, 4) if n % 2 == 0 else (444, 7, 3)
        bits, vals = tables(kind)
        qt = np.full((2, 64), step, np.uint16)
        qt[:, 1::3] = max(1, step - 1)
        levels.append([encode(blocks(rng, mx * my, 6 if sampling == 420 else 3, density, amplitude), sampling, mx, my,
                              qt, bits, vals)])
    ts = synth.TextureSet(levels)
    ctx = jt.Context(0, max_cache_blocks=1 << 10)
    ctx.set_tuning(**{**ctx.tuning(), "decode_mcus_per_warp": mcus, "decode_warps": 2, "decode_ctas_per_sm": 1})
    ctx.upload_set(ts)
    gb = mcu_grid_gbuffer(ts, 64)
    frame(ctx, jt.DeviceGBuffer.from_host(gb), 0, torch)
    ctx.stats()
    work = ctx.work_list()
    assert work.size == ts.total_mcus()
    check_tiles(ctx, oracle.texset_from(ts), GidMap(ts), work)
    ctx.close()
