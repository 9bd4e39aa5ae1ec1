"""The raster's triangle classes and work splits against the oracle's hit
IDs: one triangle to a few hundred, screen sizes on both sides of the 64-pixel
extent that the 32-bit walk takes, triangles that leave the image, depth
ranges on both sides of its limit, and meshes so small that several warps
share a triangle -- through the plain launches and the persistent batch,
which split them differently."""

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


def _fan(tris):
    """Shell of explicit triangles [T, 3, 3], UVs from the vertex index."""
    pos = np.asarray(tris, np.float32).reshape(-1, 3)
    n = len(pos)
    uv = np.stack([(np.arange(n) % 7) / 7.0, (np.arange(n) % 5) / 5.0], 1).astype(np.float32)
    return pos, uv, np.arange(n, dtype=np.int32).reshape(-1, 3)


def _both_sides(t):
    t = np.asarray(t, np.float64)
    return np.concatenate([t, t[:, [0, 2, 1]]])   # one of the two windings faces the camera


def _scene(geos):
    rng = np.random.default_rng(3)
    return Scene([Shell(p, u, t, synth.rgba_texture(32, 32, rng), FMT_RGBA_F32) for p, u, t in geos])


def _cases():
    rng = np.random.default_rng(5)
    one = _both_sides([[[0.0, -0.4, -0.3], [0.1, 0.5, -0.2], [-0.1, 0.0, 0.6]]])
    huge = _both_sides([[[0.0, -40.0, -30.0], [0.0, 50.0, -20.0], [0.0, 0.0, 60.0]]])
    # slivers that run towards the camera: narrow on the screen, 0.3 to 3.5 deep
    deep = _both_sides(np.stack([np.array([[2.7, y, -0.02], [-0.5, y + 0.02, 0.0], [2.6, y + 0.03, 0.02]])
                                 for y in np.linspace(-0.05, 0.05, 9)]))
    soup = _both_sides(rng.normal(0, 0.5, (150, 1, 3)) + rng.normal(0, 0.15, (150, 3, 3)))
    cam = dict(eye=(3.0, 0.1, 0.2))
    yield "one", [_fan(one)], dict(cam, width=65, height=63)
    yield "one_large", [_fan(one)], dict(cam, width=900, height=700)
    yield "off_screen", [_fan(huge), synth.icosphere(1, 0.8)], dict(cam, width=333, height=201)
    yield "deep", [_fan(deep), _fan(soup)], dict(cam, width=300, height=280)
    yield "soup_small", [_fan(soup)], dict(cam, width=40, height=31)
    yield "soup_large", [_fan(soup)] * 3, dict(cam, width=1200, height=900)
    yield "ico_near", [synth.icosphere(2, 1.0), synth.icosphere(0, 0.9)], dict(eye=(1.6, 0.3, 0.2), width=500, height=400)
    yield "ico_far", [synth.icosphere(3, 1.0)] * 2, dict(eye=(9.0, 0.3, 2.0), width=500, height=400)


@pytest.mark.parametrize("name,geos,cam", list(_cases()), ids=lambda v: v if isinstance(v, str) else "")
def test_raster_classes_match_oracle(vs, ctx, name, geos, cam):
    scene = _scene(geos)
    cam = synth.look_at(**cam)
    ref, ref_hits, frags = oracle.render(scene, cam)
    assert (ref_hits >= 0).any()
    obj = vs.ShellObject.from_scene(ctx, scene)
    ws = vs.make_workspace(ctx, [obj, obj], [cam, cam])
    out, hits = vs.render(ctx, obj, cam, ws)
    st = vs.read_stats(ws, reset=True)
    assert st["device_status"] == 0 and st["fragments"] == frags.sum()
    assert np.array_equal(hits.cpu().numpy(), ref_hits)
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-5
    items = [dict(obj=obj, cam=cam, out=torch.empty_like(out), hits=torch.empty_like(hits)) for _ in range(2)]
    vs.render_batch(ctx, items, ws)
    both = vs.read_stats(ws)
    assert both["device_status"] == 0
    for k in ("fragments", "tris_front", "tris_culled_back", "tris_culled_near", "tris_culled_guard", "tris_large",
              "tris_clipped"):
        assert both[k] == 2 * st[k], k
    for it in items:
        assert torch.equal(it["out"], out) and torch.equal(it["hits"], hits)
