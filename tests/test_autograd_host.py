"""The gradients that VSRender returns, with the renderer replaced by host
arithmetic: each texture's gradient stands for itself in autograd (its own
version counter, accumulation on its own), and one that is asked for alone
holds no memory of the others'."""

import ctypes
import importlib
import types

import pytest
import torch

render = importlib.import_module("paper_2409_02482_gb300.render")
SHAPES = [(3, 5, 4), (2, 7, 4), (1, 1, 4)]


@pytest.fixture
def scene(monkeypatch):
    """obj with texel and gradient pitches; gradient i is i + 1 everywhere."""

    def fake_render(vctx, obj, cam, ws, bg=None, flags=0):
        return torch.zeros(6, 8, 4), torch.zeros(obj.k, 6, 8, dtype=torch.int32)

    def fake_into(vctx, obj, cam, ws, hits, grad_rgb, ptrs, bg, loss, flags, stream):
        for i, (p, (h, w, c)) in enumerate(zip(ptrs, obj.grad_shapes())):
            a = (ctypes.c_float * (h * w * c)).from_address(p)
            for q in range(h * w * c):
                a[q] += i + 1

    monkeypatch.setattr(render, "render", fake_render)
    monkeypatch.setattr(render, "_backward_into", fake_into)

    def make(dtypes, pitch, frozen=()):
        tex = [torch.zeros(*s, dtype=d, requires_grad=i not in frozen) for i, (s, d) in enumerate(zip(SHAPES, dtypes))]
        shapes = [(h, w, pitch or c) for h, w, c in SHAPES]
        obj = types.SimpleNamespace(k=len(tex), textures=tex, grad_shapes=lambda: shapes,
                                    zero_grads=lambda: [torch.zeros(s) for s in shapes])
        return tex, lambda: render.VSRender.apply(None, obj, None, None, (0.0, 0.0, 0.0), 0, *tex)

    return make


F16, F32 = torch.float16, torch.float32
FORMS = [((F32,) * 3, None), ((F16,) * 3, None), ((F16, F32, F16), None), ((F32, F32, F16), None), ((F16,) * 3, 4),
         ((F16,) * 3, 6), ((F32,) * 3, 3)]


@pytest.mark.parametrize("dtypes,pitch", FORMS)
def test_a_gradient_changed_in_place_is_the_only_one_changed(scene, dtypes, pitch):
    tex, draw = scene(dtypes, pitch)
    g = torch.autograd.grad(draw(), tex, torch.ones(6, 8, 4))
    w = torch.full_like(g[0], 2.0, requires_grad=True)
    y = (w * g[0]).sum()          # autograd saves g[0]
    g[1].mul_(3)
    g[2].add_(1)
    y.backward()                  # refused if g[0] counted as changed with g[1]
    c = min(4, pitch or 4)
    assert torch.equal(w.grad, g[0]) and (g[0][..., :c] == 1).all() and (g[1][..., :c] == 6).all()
    assert [t.shape for t in g] == [t.shape for t in tex] and [t.dtype for t in g] == list(dtypes)


@pytest.mark.parametrize("dtypes,pitch", FORMS)
def test_accumulation_after_one_gradient_is_cleared(scene, dtypes, pitch):
    tex, draw = scene(dtypes, pitch)
    draw().sum().backward()
    tex[1].grad = None
    draw().sum().backward()
    c = min(4, pitch or 4)
    for i, n in enumerate((2, 1, 2)):
        assert (tex[i].grad[..., :c] == n * (i + 1)).all() and not tex[i].grad[..., c:].any()


@pytest.mark.parametrize("dtypes,pitch", FORMS)
def test_a_gradient_asked_for_alone_holds_its_own_memory(scene, dtypes, pitch):
    tex, draw = scene(dtypes, pitch, frozen=(0,))
    g1, g2 = torch.autograd.grad(draw(), tex[1:], torch.ones(6, 8, 4))
    for g, t, v in ((g1, tex[1], 2), (g2, tex[2], 3)):
        h, w, c = t.shape
        assert g.untyped_storage().nbytes() <= h * w * max(c, pitch or c) * 4
        assert (g[..., :min(c, pitch or c)] == v).all()
