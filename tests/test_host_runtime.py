"""Host logic of the library on a CUDA runtime of host memory (fake_runtime.cpp): decode tables,
and what the calls keep and leave behind. No GPU needed."""

import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INCLUDE = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def fake_library(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INCLUDE, "cuda_runtime.h")):
        pytest.skip("no host C++ compiler or no CUDA headers")
    import paper_2510_08166_gb300 as jt
    so = str(tmp_path_factory.mktemp("fake") / "libjt_fake.so")
    subprocess.check_call([cxx, "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CUDA_INCLUDE,
                           "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2510_08166_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "fake_runtime.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    for name, argtypes in jt._SIGS.items():
        if hasattr(lib, name):
            f = getattr(lib, name)
            f.argtypes = argtypes
            f.restype = ctypes.c_char_p if name in ("jt_last_error", "jt_status_string") else ctypes.c_int
    lib.fake_begin_capture.restype = ctypes.c_void_p
    lib.fake_scene_tables.restype = lib.fake_last_malloc.restype = lib.fake_set_bytes.restype = ctypes.c_size_t
    return lib


@pytest.fixture
def fake(fake_library, monkeypatch):
    """The package's binding over the fake library."""
    import paper_2510_08166_gb300 as jt
    monkeypatch.setattr(jt, "lib", lambda: fake_library)
    return fake_library


def spec(lengths, symbols):
    """(bits[16], vals[256]) of canonical codes of the given lengths (ascending)."""
    bits, vals = np.zeros(16, np.uint8), np.zeros(256, np.uint8)
    for l in lengths:
        bits[l - 1] += 1
    vals[:len(symbols)] = symbols
    return bits, vals


def naive_entries(bits, vals, dc):
    """Per 16-bit prefix: (code length, symbol) of T.81 Annex C's code assignment, else None."""
    out, code, k = [None] * 65536, 0, 0
    for l in range(1, 17):
        for _ in range(int(bits[l - 1])):
            s = int(vals[k])
            size = s if dc else s & 15
            valid = size <= (11 if dc else 10) and (dc or size or s in (0x00, 0xF0))
            for p in range(code << (16 - l), (code + 1) << (16 - l)):
                out[p] = (l, s) if valid else None
            code, k = code + 1, k + 1
        code <<= 1
    return out


def entry(l, s, dc):
    run, size = (0, s) if dc else (s >> 4, s & 15)
    if not dc and s == 0:
        run = 63
    return (l + size) | (size << 5) | (run << 10)


DC, AC = list(range(12)), [0x00, 0x01, 0x02, 0x11, 0x03, 0x21, 0x12, 0x31, 0xF0, 0x04, 0x41, 0x05]
SHAPES = {
    "one short, one long": [1, 16],                # 514 entries: w >> 22 alone reaches past them
    "a few short, one long": [4] * 11 + [12],
    "one long": [11],
    "short only": [4] * 12,
    "complete but for one prefix": list(range(1, 12)) + [16],
    "long only": [13] * 12,
    "every code long": [11] * 255 + [12],          # (almost) the most prefixes that long codes can take
    "half of them long": [4] * 8 + [11] * 154,
}


@pytest.mark.parametrize("name", SHAPES)
@pytest.mark.parametrize("at", [(0, 1, 2, 3), (3,), (0,)])
def test_every_prefix_finds_its_entry(fake, name, at):
    import paper_2510_08166_gb300 as jt
    std_bits, std_vals, _ = synth.standard_huffman()
    enc = synth.encode(synth.texture(1, 16, 16), 80, 420)
    lengths = SHAPES[name]
    bits, vals = std_bits.copy(), std_vals.copy()
    for t in at:
        bits[t], vals[t] = spec(lengths, np.resize(AC if t & 1 else DC, len(lengths)))
    enc.huff_bits, enc.huff_vals = bits, vals
    ctx = jt.Context(0, 64)
    ctx.upload(0, 0, enc)
    got = np.empty((1, 4, 65536), np.int32)
    fake.fake_table_entries(ctx._h, ctypes.c_void_p(got.ctypes.data))
    for t in range(4):
        want = np.array([0xFFE0 if e is None else entry(*e, t % 2 == 0) for e in naive_entries(bits[t], vals[t], t % 2 == 0)])
        assert np.array_equal(got[0, t], want), (t, np.flatnonzero(got[0, t] != want)[:4])
    ctx.close()


def device(a):
    """A host array as the fake runtime's device memory, with what the binding asks of a tensor."""
    a.data_ptr = lambda: a.ctypes.data
    return a


class Array(np.ndarray):
    """An array that can carry a data_ptr (16-byte aligned, as numpy's larger arrays are)."""


def zeros(*shape, dtype=np.float32):
    return device(np.zeros(shape, dtype).view(Array))


class GBuffer:
    def __init__(self, w, h):
        self.width, self.height = w, h
        self.uv, self.tex_id, self.mip = zeros(h, w, 2), zeros(h, w, dtype=np.uint16), zeros(h, w, dtype=np.uint8)

    def c(self):
        import paper_2510_08166_gb300 as jt
        return jt.jt_gbuffer(self.uv.data_ptr(), self.tex_id.data_ptr(), self.mip.data_ptr(), self.width, self.height)


def test_a_failed_float_pass_leaves_no_counts_to_the_next(fake):
    import paper_2510_08166_gb300 as jt
    ctx = jt.Context(0, 1 << 10)
    ctx.register_coeff_textures(0, 1, 64, 64)
    gb, coef, out = GBuffer(64, 16), zeros(1, 4, 4, 6, 64), zeros(16, 64, 3)
    for _ in range(2):
        ctx.colorize_float(gb, coef, out, 0)
    for run in (lambda: ctx.colorize_float(gb, coef, out, 0), lambda: ctx.colorize_backward(gb, out, coef, 0)):
        fake.fake_fail_gather(1)
        with pytest.raises(jt.JTError):
            run()
        fake.fake_fail_gather(0)
        # a pass that is only captured clears nothing: the eager one after it still has to
        fake.fake_begin_capture()
        run()
        fake.fake_end_capture()
        run()
        run()
        ctx.stats()
        assert not fake.fake_cursors_dirty()
    ctx.close()


class Scene:
    """What raster_scene takes: `n` textures of sides of their own and three quads."""

    def __init__(self, seed, n):
        self.width = self.height = 16
        self.cam, self.rot = [0, 1, 0], [1, 0, 0, 0, 1, 0, 0, 0, 1]
        self.ax = self.ay = self.tan_x = self.tan_y = self.max_t = self.kx = self.ky = 1.0
        self.shift, self.cell_seed, self.use_mips = 0.0, 1, 1
        self.tex_w = np.arange(1, n + 1, dtype=np.int32) + seed * 1000
        self.tex_h, self.tex_levels = self.tex_w + 5, np.full(n, 1 + seed % 4, np.int32)
        self.quads = np.zeros(3, synth.QUAD_DTYPE)
        self.quads["tex"], self.quads["rep"] = np.arange(3) % n, seed

    def tables(self):
        t = np.zeros((len(self.tex_w), 4), np.float32)
        t[:, 0], t[:, 1], t[:, 2] = self.tex_w, self.tex_h, self.tex_levels.view(np.float32)
        return t.tobytes() + self.quads.tobytes()


def scene_tables(fake):
    out = np.zeros(fake.fake_scene_tables(None), np.uint8)
    fake.fake_scene_tables(ctypes.c_void_p(out.ctypes.data))
    return out.tobytes()


def test_a_scene_is_copied_from_memory_that_outlives_the_call(fake):
    import paper_2510_08166_gb300 as jt
    ctx, gb = jt.Context(0, 64), GBuffer(16, 16)
    for seed in range(40):  # more calls than the host memory has turns, the copies read late
        s = Scene(seed, 1 + seed * 7 % 50)
        ctx.raster_scene(s, gb, 0)
        if seed % 3 == 0:
            assert scene_tables(fake) == s.tables()
    assert scene_tables(fake) == s.tables()
    ctx.close()


def test_a_captured_scene_keeps_its_tables(fake):
    import paper_2510_08166_gb300 as jt
    ctx, gb = jt.Context(0, 64), GBuffer(16, 16)
    ctx.raster_scene(Scene(0, 9), gb, 0)
    graph = fake.fake_begin_capture()
    s = Scene(1, 9)
    ctx.raster_scene(s, gb, 0)
    fake.fake_end_capture()
    for seed in range(2, 30):  # others come between its launches, larger ones too
        other = Scene(seed, 9 if seed < 20 else 400)
        ctx.raster_scene(other, gb, 0)
        assert scene_tables(fake) == other.tables()
        fake.fake_launch_graph(ctypes.c_void_p(graph))
        assert scene_tables(fake) == s.tables()
    assert fake.fake_owned(ctypes.c_void_p(graph)) == 1
    fake.fake_destroy_graph(ctypes.c_void_p(graph))
    assert fake.fake_owned(ctypes.c_void_p(graph)) == 0
    ctx.close()


@pytest.mark.parametrize("mcus,warps", [(16, 14), (32, 7), (8, 9), (4, 1)])  # the default, a listed one, two of neither
def test_autotune_times_the_shape_in_use(fake, mcus, warps):
    import paper_2510_08166_gb300 as jt
    ctx, gb, out = jt.Context(0, 64), GBuffer(64, 64), zeros(64, 64, 4, dtype=np.uint8)
    ctx.upload(0, 0, synth.encode(synth.texture(1, 64, 64), 80, 420))
    used = {**ctx.tuning(), "decode_mcus_per_warp": mcus, "decode_warps": warps, "decode_ctas_per_sm": 1}
    ctx.set_tuning(**used)
    fake.fake_fast_shape(mcus, warps)
    best, ms = ctx.autotune([(gb, out)], jt.FILTER_BILINEAR, reps=2, stream=0)
    assert ms == 1.0 and (best["decode_mcus_per_warp"], best["decode_warps"]) == (mcus, warps)
    # the default is found from any other shape too
    fake.fake_fast_shape(16, 14)
    best, ms = ctx.autotune([(gb, out)], jt.FILTER_BILINEAR, reps=2, stream=0)
    assert ms == 1.0 and (best["decode_mcus_per_warp"], best["decode_warps"]) == (16, 14)
    ctx.close()


@pytest.mark.parametrize("sms", [40, 152])
def test_tiles_go_by_the_device_s_sm_count(fake, sms):
    import paper_2510_08166_gb300 as jt
    fake.fake_sm_count(sms)
    try:
        ctx = jt.Context(0, 64)
    finally:
        fake.fake_sm_count(152)
    ctx.upload(0, 0, synth.encode(synth.texture(1, 64, 64), 80, 420))
    for tiles in (4 * sms - 1, 4 * sms, 8 * sms - 1, 8 * sms):  # high tiles of 128 x 32 pixels in a column
        gb = GBuffer.__new__(GBuffer)
        one = zeros(16)
        gb.uv = gb.tex_id = gb.mip = one
        gb.width, gb.height = 128, 32 * tiles
        ctx.mark(gb, jt.FILTER_NEAREST, 0)
        assert fake.fake_tile_h() == (8 if tiles < 4 * sms else 32)
        assert fake.fake_many() == (tiles >= 8 * sms)
        ctx.decode(0)
        s = Scene(1, 2)
        s.width, s.height = gb.width, gb.height = 1024, 2 * tiles
        ctx.raster_scene(s, gb, 0)
        rows = -(-2 * tiles // 8)
        assert fake.fake_tile_x() == next(x for x in (256, 128, 64, 32) if x == 32 or 1024 // x * rows >= 8 * sms)
    ctx.close()


def test_the_bench_counts_the_bucket_that_the_library_allocates(fake, monkeypatch):
    import paper_2510_08166_gb300 as jt
    monkeypatch.syspath_prepend(ROOT)
    import bench
    ctx = jt.Context(0, 1 << 10)
    ctx.register_coeff_textures(0, 1, 64, 64)
    ctx.colorize_float(GBuffer(64, 16), zeros(1, 4, 4, 6, 64), zeros(16, 64, 3), 0)
    assert bench.bucket_bytes(64 * 16) == 2 * fake.fake_last_malloc()  # written once and read once
    ctx.close()


def test_an_upload_after_one_that_ran_out_of_memory_has_its_tables(fake):
    import paper_2510_08166_gb300 as jt
    ctx, gb = jt.Context(0, 64), GBuffer(64, 64)
    encs = [synth.encode(synth.texture(1, 64, 64), q, 420) for q in (80, 50)]
    encs[1].huff_bits, encs[1].huff_vals = encs[1].huff_bits.copy(), encs[1].huff_vals.copy()
    encs[1].huff_bits[0], encs[1].huff_vals[0] = spec([4] * 12, DC)
    ctx.upload(0, 0, encs[0])
    fake.fake_fail_malloc(ctypes.c_size_t(fake.fake_set_bytes()))  # the tables grow for the second set
    with pytest.raises(jt.JTError):
        ctx.upload(1, 0, encs[1])
    for t in range(2):  # the first texture is as it was, and the second one can be uploaded again
        ctx.mark(gb, jt.FILTER_NEAREST, 0)
        ctx.decode(0)
        assert fake.fake_tables_on_device() == t + 1
        ctx.upload(1 + t, 0, encs[1])
    ctx.close()
