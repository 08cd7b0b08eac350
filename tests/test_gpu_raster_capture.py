"""A captured jt_raster_scene: its launches rasterise its own scene, whatever other scenes, larger
ones too, the context has taken since and whatever became of the caller's arrays."""

import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SIZES = [(1024, 1024), (2048, 2048), (512, 512), (4096, 4096)]


def scene(seed, nquads):
    return synth.scene_desc(seed, 320, 180, SIZES, [11, 12, 10, 13], synth.Pose(quad_seed=seed), nquads=nquads)


def planes(gb):
    return [t.clone() for t in (gb.uv, gb.tex_id, gb.mip)]


def test_captured_scene():
    import paper_2510_08166_gb300 as jt
    ctx, gb, other = jt.Context(0, max_cache_blocks=64), jt.DeviceGBuffer.empty(320, 180), jt.DeviceGBuffer.empty(320, 180)
    ctx.raster_scene(scene(5, 60), gb)
    torch.cuda.synchronize()
    want = planes(gb)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.raster_scene(scene(5, 60), gb)
    for n in (60, 40, 900, 4000):
        ctx.raster_scene(scene(7, n), other)
        for t in (gb.uv, gb.tex_id, gb.mip):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(planes(gb), want))
        ctx.raster_scene(scene(7, n), gb)
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(planes(gb), planes(other)))
    del graph
    ctx.close()
