"""GPU rasteriser against the oracle where its forms change: rolled and level cameras, one texture
and counts around powers of two (the remainder by a reciprocal), tile widths and ragged
edges, more quads in a tile than are staged, footprints beyond the last level."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("W,H,ntex,nquads,roll,cam", [
    (257, 9, 1, 0, 0.0, (0.0, 1.7, 0.0)),
    (31, 8, 2, 3, 0.0, (5.0, 0.3, -2.0)),
    (640, 361, 3, 400, 0.2, (1.0, 1.7, 2.0)),
    (300, 200, 255, 1500, 0.0, (0.0, 40.0, 0.0)),
    (1920, 1080, 257, 200, 0.0, (-3.0, 1.7, 1.0)),
    (700, 500, 65535, 64, -0.4, (2e6, 9.0, -3e6)),
])
def test_forms(W, H, ntex, nquads, roll, cam):
    import paper_2510_08166_gb300 as jt
    sizes = [(1 << (i % 13), 1 << (i % 12)) for i in range(ntex)]
    levels = [1 + i % 13 for i in range(ntex)]
    d = synth.scene_desc(11, W, H, sizes, levels, synth.Pose(cam, 30.0, -15.0, 70.0, 5, 0.0), nquads=nquads)
    if roll:
        c, s = np.cos(roll), np.sin(roll)
        r = d.rot.reshape(3, 3).astype(np.float64) @ np.array([[c, -s, 0], [s, c, 0], [0, 0, 1]])
        d.rot = r.astype(np.float32).reshape(-1)
    ctx = jt.Context(0, max_cache_blocks=16)
    gb = jt.DeviceGBuffer.empty(W, H)
    ctx.raster_scene(d, gb)
    uv, tex, mip = oracle.raster_scene(d)
    np.testing.assert_array_equal(gb.tex_id.cpu().numpy().view(np.uint16), tex)
    np.testing.assert_array_equal(gb.mip.cpu().numpy(), mip)
    np.testing.assert_array_equal(gb.uv.cpu().numpy().view(np.uint32), uv.view(np.uint32))
    ctx.close()
