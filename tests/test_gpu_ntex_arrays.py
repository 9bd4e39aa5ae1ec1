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


CHUNK = 1 << 18   # texels that a workspace is sized for


@pytest.mark.parametrize("levels,features,hidden,out_ch,W,H,fused", [
    (16, 2, 4, 1, 1501, 799, True),      # an odd last chunk: dX in single values
    (16, 4, 5, 1, 1501, 799, True),
    (16, 3, 5, 2, 1501, 799, True),
    (16, 4, 64, 4, 1501, 1201, True),
    (8, 2, 65, 5, 1501, 799, False),     # more hidden units than the fused kernels take
    (8, 4, 64, 33, 1501, 799, False),    # more outputs than the fused adjoint takes
])
def test_fp32_chunks_end_inside_a_texel_row(vs, ctx, levels, features, hidden, out_ch, W, H, fused):
    """FP32 networks whose adjoint runs in several chunks of texels that end
    inside a texel row: the fused kernel's chunks fill the workspace with dX
    alone, the layers' own hold every activation of 2^18 texels.  Texels and
    the gradient of sampled texels, among them those around each chunk's end,
    against the oracle at the FP32 bars of its other tests (1e-4 of the
    largest value).  Texels with a hidden unit within 1e-4 of zero, whose ReLU
    mask FP32 rounding could turn, get no gradient."""
    cfg = ntex.NtexConfig(levels=levels, features=features, log2_table=10, base_res=4, growth=1.25, hidden=hidden,
                          out_ch=out_ch)
    nt, params = _net(vs, ctx, cfg, W, H, 21)
    N, LF = W * H, levels * features
    size = CHUNK
    if fused:
        most = (nt.ws.numel() // 4 - 64) // LF
        size = -(-N // -(-N // most))
        size = min(-(-size // 64) * 64, most)
    ends = list(range(size, N, size))
    assert ends and all(e % W for e in ends)
    rng = np.random.default_rng(22)
    idx = np.unique(np.concatenate([rng.choice(N, 3000, replace=False), [0, N - 1]] +
                                   [np.arange(e - 40, e + 40) for e in ends]))
    P = ntex.unpack(cfg, params)
    y, a = ntex._mlp(cfg, P, ntex.texel_centres(W, H)[idx])
    tex = torch.zeros(H, W, out_ch, device="cuda")
    nt.forward(tex)
    got = tex.reshape(-1, out_ch).cpu().numpy()[idx]
    assert np.abs(got - y).max() <= 1e-4 * max(1.0, np.abs(y).max())
    g = rng.normal(size=(len(idx), out_ch)).astype(np.float32)
    g[np.minimum(np.abs(a["z1"]).min(1), np.abs(a["z2"]).min(1)) < 1e-4] = 0.0
    assert (np.abs(g).max(1) > 0).mean() > 0.9
    dense = torch.zeros(N, out_ch, device="cuda")
    dense[torch.from_numpy(idx).cuda()] = torch.from_numpy(g).cuda()
    nt.backward(dense.reshape(H, W, out_ch))
    ref = ntex.backward(cfg, params, W, H, g.astype(np.float64), texels=idx)
    q = nt.grads.cpu().numpy()
    for name, off, shp in cfg.layout()[0]:
        m = int(np.prod(shp))
        r = ref[off:off + m]
        assert np.abs(r).max() > 0 and np.abs(q[off:off + m] - r).max() <= 1e-4 * np.abs(r).max(), name
    assert nt.status() == 0
