"""The FP32 form where a call's pairs are taken in more than one group or range: bit-equal to the pairs
taken one by one, since a pair's own sums do not depend on the others and the pairs are added in order."""
import pytest
import torch

from paper_2305_11566_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fp32", "bf16"])
@pytest.mark.parametrize("n,W,H", [(96, 256, 128), (60, 131, 77)], ids=["slots", "odd"])
def test_gradients_of_many_pairs(svlib, form, n, W, H):
    """96 crops of 256 x 128, 32/64/128 net: 1.8 GB of slots for dec2, two ranges of at most 1 GiB.  And odd
    crops; a pair alone also takes the input gradients' form for launches that leave SMs idle."""
    shape, D = synth.NET_WIDE, 16
    g = torch.Generator(device="cuda").manual_seed(3)
    f32 = {"device": "cuda", "dtype": torch.float32, "generator": g}
    ctx = binding.Context(shape, 7, form)
    try:
        ctx.set_weights(synth.he_normal_weights(shape, 7))
        dp = binding.to_device(synth.make_pair(W, H, 40.0, 5), D)
        h3, w3 = binding.latent_hw(H, W)
        coarse = [torch.rand(H // 4, W // 4, **f32) * (D - 1) for _ in range(n)]
        eps = [torch.randn(h3, w3, shape.latent, **f32) for _ in range(n)]
        gY = [torch.randn(H, W, **f32) * 1e-4 for _ in range(n)]
        gl = [torch.randn(h3, w3, shape.latent, **f32) * 1e-5 for _ in range(n)]
        ctx.refine_train([dp] * n, coarse, eps)
        many, many_c = ctx.refine_backward(gY, gl, gl, True, coarse)
        total = torch.zeros_like(many)
        for i in range(n):
            ctx.refine_train([dp], coarse[i:i + 1], eps[i:i + 1])
            one, one_c = ctx.refine_backward(gY[i:i + 1], gl[i:i + 1], gl[i:i + 1], True, coarse[i:i + 1])
            total += one
            assert torch.equal(many_c[i], one_c[0])
        ctx.synchronize()
        assert many.abs().max() > 0 and torch.equal(many, total)
    finally:
        ctx.close()


def test_refine_around_a_group_boundary(svlib):
    """A 1242 x 375 pair of the 32/64/128 net has 134.4 MB of activations, so 2 GiB hold 15: pairs 14 and 15
    of a call are the last of one group and the first of the next."""
    shape, W, H, D, n = synth.NET_WIDE, 1242, 375, 48, 17
    g = torch.Generator(device="cuda").manual_seed(4)
    ctx = binding.Context(shape, 9, "fp32")
    try:
        ctx.set_weights(synth.he_normal_weights(shape, 7))
        dp = binding.to_device(synth.make_pair(W, H, 190.0, 5), D)
        maps = [torch.randint(0, D, (H // 4, W // 4), device="cuda", generator=g, dtype=torch.int16) for _ in range(n)]
        many = ctx.refine([dp] * n, maps)
        for i in (13, 14, 15, 16):
            assert torch.equal(many[i], ctx.refine([dp], [maps[i]])[0])
        ctx.synchronize()
    finally:
        ctx.close()
