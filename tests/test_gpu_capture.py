"""Calls captured into a caller's own CUDA graph, after a call of the same sizes has allocated the
workspaces: a replay on new inputs gives what the same calls give eagerly, bit for bit."""
import pytest
import torch

from paper_2305_11566_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fp32", "bf16", "table1"])
def test_replay_equals_eager(svlib, form):
    sizes, D = [(131, 66), (64, 48), (97, 101)], 6
    t1 = form == "table1"
    shape = form if t1 else synth.NET_SMALL
    g = torch.Generator(device="cuda").manual_seed(1)
    f32 = {"device": "cuda", "dtype": torch.float32}
    ctx = binding.Context(shape, 3, "fp32" if t1 else form)
    try:
        ctx.set_weights(torch.randn(ctx.n_params, **f32, generator=g) * 0.05)
        dps = [binding.to_device(synth.make_pair(W, H, 20.0, 3 + W), D) for W, H in sizes]
        maps = [torch.empty(H // 4, W // 4, device="cuda", dtype=torch.int16) for W, H in sizes]
        coarse = [torch.empty(H // 4, W // 4, **f32) for W, H in sizes]
        eps = [torch.empty(*binding.latent_hw(H, W), ctx.latent, **f32) for W, H in sizes]
        gt = [torch.empty(H, W, **f32) for W, H in sizes]

        def fresh():
            for m, c, e, t in zip(maps, coarse, eps, gt):
                m.copy_(torch.randint(0, D, m.shape, device="cuda", generator=g))
                c.copy_(torch.rand(c.shape, **f32, generator=g) * (D - 1))
                e.copy_(torch.randn(e.shape, **f32, generator=g))
                t.copy_(torch.rand(t.shape, **f32, generator=g) * 20)

        def calls():
            out = list(ctx.refine(dps, maps)) if form != "bf16" else []
            Y, mu, lv = ctx.refine_train(dps, coarse, eps)
            out += [*Y, *mu, *lv]
            if not t1:
                loss, gY, gmu, glv = ctx.loss(dps, Y, gt, mu, lv)
                grad, gc = ctx.refine_backward(gY, gmu, glv, True, coarse)
                out += [loss, *gY, grad, *gc]
            return out

        fresh()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            calls()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            held = calls()
        junk = [bytearray(64 * i) for i in range(1, 400)]  # other owners of the host memory the calls freed
        for _ in range(2):
            fresh()
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
            got = [t.clone() for t in held]
            want = calls()
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(got, want))
            assert any(bool(t.abs().sum() > 0) for t in got)
        del junk
        ctx.synchronize()
    finally:
        ctx.close()
