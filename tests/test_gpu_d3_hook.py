"""sv_debug_activation of d3 after calls that ran the fused decoder tail: refused where every output width is
even, made from the call's d2 where one is odd."""
import numpy as np
import pytest
import torch

from paper_2305_11566_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["bf16", "fp8"])
def test_d3_after_a_fused_call(svlib, form):
    shape, sizes, D = synth.NET_WIDE, [(255, 66), (132, 75), (97, 49)], 6
    ctx = binding.Context(shape, 5, form)
    try:
        ctx.set_weights(synth.he_normal_weights(shape, 7))
        dps = [binding.to_device(synth.make_pair(W, H, 20.0, 3 + W), D) for W, H in sizes]
        stream = torch.cuda.Stream()

        def d3(i):
            return ctx.debug_activation(6, i, (sizes[i][1], sizes[i][0], shape.dec[2]))
        maps = ctx.coarse_match(dps)
        ctx.set_option("fused_final", 0)
        ctx.refine(dps, maps)
        torch.cuda.synchronize()
        want = [d3(i) for i in range(3)]
        ctx.set_option("fused_final", 1)
        Y = ctx.refine(dps, maps)
        torch.cuda.synchronize()
        got = [d3(i) for i in range(3)]
        assert all(np.array_equal(a, b) for a, b in zip(got, want)) and any(a.any() for a in got)
        for _ in range(3):  # captured, then replayed
            out = ctx.pipeline(dps, stream=stream)
            stream.synchronize()
            ctx.pipeline(dps[1:2], stream=stream)  # an even width alone
            stream.synchronize()
            with pytest.raises(binding.SvError):
                ctx.debug_activation(6, 0, (sizes[1][1], sizes[1][0], shape.dec[2]))
            again = ctx.pipeline(dps, stream=stream, out=out)
            stream.synchronize()
            assert np.array_equal(d3(2), want[2]) and np.array_equal(d3(0), want[0])
            assert all(torch.equal(a, b) for a, b in zip(again, Y))
        ctx.synchronize()
    finally:
        ctx.close()
