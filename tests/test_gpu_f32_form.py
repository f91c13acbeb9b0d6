"""GPU parity of the batched FP32 form at the sizes where its tiles can go wrong.

Level sizes just below, at and above the 16 / 32-wide tiles, odd crops in either direction (the
edge form of the nearest-x2 layers), widths that take every output-channel block (8, 4, 2
groups of 8 channels), mixed sizes in one call and more than one group of pairs.  Bar: the
FP32 form's 1e-4 px against the FP64 oracle on every pixel (a 46 k-term FP32 sum of O(1)
products stays below 1e-5 px here; the output itself is rounded at |Y| < 256 to 1.5e-5)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_11566_gb300 import binding, synth

pytestmark = pytest.mark.gpu

TOL_PX = 1e-4
ODD = synth.NetShape((16, 48, 32), 16, (80, 16, 48))
WIDE = synth.NetShape((64, 32, 16), 64, (128, 64, 16))


def refine(shape, sizes, k=3, D=4):
    params = synth.he_normal_weights(shape, 7)
    rng = np.random.default_rng(11)
    params += (rng.normal(size=params.size) * 0.01).astype(np.float32)  # non-zero biases
    ctx = binding.Context(shape, k, "fp32")
    try:
        ctx.set_weights(params)
        pairs = [synth.make_pair(W, H, 12.0, 70 + W + H) for W, H in sizes]
        coarse = [rng.integers(0, D, (H // 4, W // 4)).astype(np.int16) for W, H in sizes]
        dps = [binding.to_device(p, D) for p in pairs]
        got = ctx.refine(dps, [torch.from_numpy(c).cuda() for c in coarse])
        ctx.synchronize()
        for p, c, Y in zip(pairs, coarse, got):
            ref = oracle.refine_forward(shape, params, p.left, c.astype(np.float64))["Y"]
            err = np.abs(Y.cpu().numpy().astype(np.float64) - ref).max()
            assert err <= TOL_PX, f"{p.width}x{p.height}: {err:.3g}"
    finally:
        ctx.close()


@pytest.mark.parametrize("W,H", [(16, 16), (17, 19), (31, 33), (64, 64), (63, 66), (65, 63), (127, 30), (130, 129),
                                 (258, 35)])
@pytest.mark.parametrize("shape", [synth.NET_SMALL, ODD, WIDE], ids=["small", "odd", "wide"])
def test_refine_edges_of_tiles(svlib, shape, W, H):
    refine(shape, [(W, H)])


def test_refine_mixed_sizes_in_one_call(svlib):
    refine(ODD, [(64, 33), (19, 40), (131, 66), (16, 16), (97, 64)])


def test_refine_more_than_one_group(svlib):
    """20 frames of the widest net exceed the activation budget of one group; the last pair of a
    later group equals the same pair refined alone."""
    shape, k, D, W, H = synth.NET_WIDE, 9, 48, 1242, 375
    ctx = binding.Context(shape, k, "fp32")
    try:
        ctx.set_weights(synth.he_normal_weights(shape, 7))
        dp = binding.to_device(synth.make_pair(W, H, 190.0, 5), D)
        rng = np.random.default_rng(2)
        maps = [torch.from_numpy(rng.integers(0, D, (H // 4, W // 4)).astype(np.int16)).cuda() for _ in range(20)]
        many = ctx.refine([dp] * 20, maps)
        for i in (0, 15, 16, 19):
            assert torch.equal(many[i], ctx.refine([dp], [maps[i]])[0])
        ctx.synchronize()
    finally:
        ctx.close()


@pytest.mark.parametrize("shape,sizes", [
    (synth.NET_SMALL, [(16, 16), (33, 17), (64, 64)]),
    (ODD, [(31, 35), (66, 63), (130, 40)]),
    (WIDE, [(129, 67)]),
    (synth.NetShape((32, 16, 48), 32, (16, 32, 80)), [(61, 30), (40, 59)]),
], ids=["small", "odd", "wide", "other"])
def test_training_gradients_edges_of_tiles(svlib, shape, sizes, k=3, D=4):
    """Weight, bias and coarse-map gradients against the FP64 oracle: 1e-4 of each layer's largest
    entry (the FP32 backward's bar), with the loss's own latent terms and caller buffers at
    4-byte alignment."""
    params = synth.he_normal_weights(shape, 7)
    rng = np.random.default_rng(12)
    params += (rng.normal(size=params.size) * 0.01).astype(np.float32)
    ctx = binding.Context(shape, k, "fp32")
    try:
        ctx.set_weights(params)
        pairs = [synth.make_pair(W, H, 12.0, 90 + W + H) for W, H in sizes]
        dps = [binding.to_device(p, D) for p in pairs]

        def odd(a):  # a copy whose base is only 4-byte aligned
            t = torch.empty(a.numel() + 1, device="cuda", dtype=a.dtype)[1:].view(a.shape)
            return t.copy_(a)
        coarse = [rng.uniform(0, D - 1, (H // 4, W // 4)) for W, H in sizes]
        eps = [rng.normal(size=(*binding.latent_hw(H, W), shape.latent)).astype(np.float32) for W, H in sizes]
        cs = [odd(torch.from_numpy(c).float().cuda()) for c in coarse]
        es = [odd(torch.from_numpy(e).cuda()) for e in eps]
        Y, mu, lv = ctx.refine_train(dps, cs, es)
        _, gY, gmu, glv = ctx.loss(dps, Y, [torch.from_numpy(p.gt).cuda() for p in pairs], mu, lv, 1e-3)
        gp, gc = ctx.refine_backward([odd(t) for t in gY], [odd(t) for t in gmu], [odd(t) for t in glv], True, cs)
        again, _ = ctx.refine_backward(gY, gmu, glv, False, cs)
        ctx.synchronize()
        assert torch.equal(gp, again)  # fixed summation order
        n_px = sum(W * H for W, H in sizes)
        n_lat = sum(e.size for e in eps)
        go = np.zeros(params.size)
        for p, c, e, g in zip(pairs, coarse, eps, gc):
            c32 = c.astype(np.float32).astype(np.float64)
            _, gi, gci = oracle.refine_backward(shape, params, p.left, c32, e.ravel(), p.gt, n_px, n_lat, 1e-3, True)
            go += gi
            assert np.abs(g.cpu().numpy() - gci).max() <= 1e-4 * np.abs(gci).max()
        got = gp.cpu().numpy()
        for name, (ow, wshape, ob, co) in oracle.param_slices(shape).items():
            n = int(np.prod(wshape))
            for o, m in ((ow, n), (ob, co)):
                ref = go[o:o + m]
                assert np.abs(got[o:o + m] - ref).max() <= 1e-4 * np.abs(ref).max() + 1e-12, (name, o == ob)
    finally:
        ctx.close()
