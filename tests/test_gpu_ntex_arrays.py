"""Neural textures on arrays that start off the boundaries of vector accesses,
and textures whose passes are cut into chunks inside a texel row."""

import ctypes

import numpy as np
import pytest
import torch

import synth
from oracle import ntex

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


def _net(vs, ctx, cfg, W, H, seed, tensor_cores=False):
    params = synth.ntex_init(cfg.shapes(), np.random.default_rng(seed))
    _, off, shp = cfg.layout()[0][0]
    n = int(np.prod(shp))
    params[off:off + n] = np.random.default_rng(seed + 1).normal(0, 0.5, n)
    nt = vs.NeuralTexture(ctx, cfg.levels, cfg.features, cfg.log2_table, cfg.base_res, cfg.growth, cfg.hidden,
                          cfg.out_ch, tex_w=W, tex_h=H, tensor_cores=tensor_cores)
    nt.params.copy_(torch.from_numpy(params))
    return nt, params.astype(np.float64)


@pytest.mark.parametrize("tensor_cores", [False, True])
@pytest.mark.parametrize("hidden", [64, 70])            # fused, and layer by layer
@pytest.mark.parametrize("levels,features", [(9, 1), (8, 2), (4, 4), (3, 8)])
def test_parameters_off_their_vector_alignment(vs, ctx, levels, features, hidden, tensor_cores):
    """params, grads and texels need 4-byte alignment only: parameter and
    gradient vectors 4, 8 and 12 bytes off a 16-byte boundary give the texels
    of an aligned network bit for bit (the same sums) and its gradients to
    the FP32 bar of the oracle's tests (the atomics' order), and leave the
    words around them alone.  Pairs of features off their boundary take the
    TF32 network from the fused kernels to the layers' own, whose FP32 sums
    run in another order: there the bars of the TF32 mode hold."""
    cfg = ntex.NtexConfig(levels=levels, features=features, log2_table=8, base_res=3, growth=1.4, hidden=hidden,
                          out_ch=9)
    W, H = 70, 50
    nt, _ = _net(vs, ctx, cfg, W, H, 3, tensor_cores)
    g = torch.randn(H, W, 12, device="cuda", generator=torch.Generator("cuda").manual_seed(4))
    ref = torch.zeros(H, W, 12, device="cuda")
    nt.forward(ref)
    nt.backward(g)
    aligned, n = nt.grads, nt.count
    params = nt.params.clone()
    for shift in (1, 2, 3):
        flat = torch.full((2, n + 8), 5.0, device="cuda")
        flat[0, shift:shift + n] = params
        flat[1, shift:shift + n] = 0.0
        nt.params, nt.grads = flat[0, shift:shift + n], flat[1, shift:shift + n]
        tex = torch.zeros_like(ref)
        nt.forward(tex)
        nt.backward(g)
        other = tensor_cores and features == 2 and hidden == 64 and shift % 2
        if other:
            assert (tex - ref).norm().item() <= 2e-3 * ref.norm().item()
        else:
            assert torch.equal(tex, ref)
        for name, off, shp in cfg.layout()[0]:
            m = int(np.prod(shp))
            r, q = aligned[off:off + m], nt.grads[off:off + m]
            if other:
                assert (q - r).norm().item() <= (1e-5 if name == "b2" else 8e-2) * r.norm().item(), name
            else:
                assert (q - r).abs().max().item() <= 1e-4 * max(r.abs().max().item(), 1e-30), name
        assert (flat[:, :shift] == 5.0).all() and (flat[:, shift + n:] == 5.0).all()
    assert nt.status() == 0
