"""Work units of the renderer's phases: image sizes and meshes at which the
last setup, clearing, raster or shading unit is partial, in a workspace whose
words are stale, through the plain launches and the persistent batch (the
sizes of its units depend on the item's place in the batch), against the
oracle's hit IDs."""

import numpy as np
import pytest
import torch

import oracle
import synth
from synth import FMT_RGBA_F32, Scene, Shell

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vs():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2409_02482_gb300 as vs
    return vs


@pytest.fixture(scope="module")
def ctx(vs):
    return vs.Context(0)


def _object(vs, ctx, subdivs):
    rng = np.random.default_rng(4)
    shells = [Shell(*synth.icosphere(s, 1.0 - 0.05 * i), synth.rgba_texture(16, 24, rng), FMT_RGBA_F32)
              for i, s in enumerate(subdivs)]
    scene = Scene(shells)
    return scene, vs.ShellObject.from_scene(ctx, scene)


@pytest.mark.parametrize("subdivs,width,height", [((0,), 31, 33), ((2, 0), 127, 65), ((3,), 1, 1),
                                                  ((5, 1, 3), 641, 359), ((6,), 257, 255)])
def test_units_cover_every_word_vertex_and_pixel(vs, ctx, subdivs, width, height):
    scene, obj = _object(vs, ctx, subdivs)
    cams = [synth.look_at((3.0, 0.2 * j, 0.3), width=width, height=height) for j in range(3)]
    ws = vs.make_workspace(ctx, [obj] * 3, cams)
    refs = [oracle.render(scene, c) for c in cams]
    for c, (ref, ref_hits, _) in zip(cams, refs):
        ws[256:].fill_(0xFF)   # behind the header: words of an earlier call
        out, hits = vs.render(ctx, obj, c, ws)
        assert np.array_equal(hits.cpu().numpy(), ref_hits)
        assert np.abs(out.cpu().numpy() - ref).max() <= 1e-5
    ws[256:].fill_(0xFF)
    items = [dict(obj=obj, cam=c, out=torch.empty(height, width, 4, device="cuda"),
                  hits=torch.empty(obj.k, height, width, dtype=torch.int32, device="cuda")) for c in cams]
    vs.render_batch(ctx, items, ws)
    st = vs.read_stats(ws)
    assert st["device_status"] == 0 and st["fragments"] == 2 * sum(int(f.sum()) for _, _, f in refs)
    for it, (ref, ref_hits, _) in zip(items, refs):
        assert np.array_equal(it["hits"].cpu().numpy(), ref_hits)
        assert np.abs(it["out"].cpu().numpy() - ref).max() <= 1e-5
