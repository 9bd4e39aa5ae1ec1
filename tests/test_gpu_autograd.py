"""VSRender's gradients against vs_render_backward on separate arrays: texel
sizes and pitches at which a shell's part of the shared buffer ends off a
16-byte boundary, gradient pitches other than the texel pitch, and shells of
different dtypes in one object."""

import numpy as np
import pytest
import torch

import synth
from synth import FMT_RGBA_F32, FMT_SH_F16, Scene, Shell

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degrees,pitch,grad_pitch", [
    ((0, 0), None, None), ((1, 1, 1), None, None), ((1, 1), 16, "tight"), ((2,), 32, 40), ((3, 3), None, None),
    ((-1, -1), None, None), ((-1, 1), None, None),   # -1: RGBA FP32
])
def test_gradients_match_separate_arrays(degrees, pitch, grad_pitch):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2409_02482_gb300 as vs
    ctx = vs.Context(0)
    rng = np.random.default_rng(6)
    shells = []
    for i, d in enumerate(degrees):
        geo = synth.icosphere(2, 1.0 - 0.05 * i)
        if d < 0:
            shells.append(Shell(*geo, synth.rgba_texture(7, 5, rng), FMT_RGBA_F32))
        else:
            c = synth.sh_channels(d)
            tex = np.zeros((7, 5, pitch or c), np.float16)
            tex[..., :c] = rng.normal(0, 0.3, (7, 5, c))
            shells.append(Shell(*geo, tex, FMT_SH_F16, d))
    obj = vs.ShellObject.from_scene(ctx, Scene(shells), grad_pitch=grad_pitch)
    cam = synth.look_at((3.0, 0.3, 0.4), width=77, height=61)
    ws = vs.make_workspace(ctx, [obj], [cam])
    tex = [t.requires_grad_() for t in obj.textures]
    out = vs.VSRender.apply(ctx, obj, cam, ws, (0.1, 0.2, 0.3), 0, *tex)
    up = torch.randn(out.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    got = torch.autograd.grad(out, tex, up)
    _, hits = vs.render(ctx, obj, cam, ws, bg=(0.1, 0.2, 0.3))
    ref = vs.render_backward(ctx, obj, cam, ws, hits, up[..., :3].contiguous(), bg=(0.1, 0.2, 0.3))
    assert vs.read_stats(ws)["device_status"] == 0
    for t, g, r in zip(tex, got, ref):
        assert g.dtype == t.dtype and g.shape == t.shape
        p = min(t.shape[2], r.shape[2])
        # the order of the FP32 atomics, then one rounding to the texels' dtype
        bar = (1e-5 + (2.0 ** -10 if t.dtype == torch.float16 else 0.0)) * r.abs().max().item()
        assert (g[..., :p].float() - r[..., :p]).abs().max().item() <= bar
        assert not g[..., p:].any()
