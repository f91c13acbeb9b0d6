"""The matcher's two job shapes and two ways of passing pairs, and the border recompute on warp MMA.

A call whose large jobs would leave SMs idle runs small jobs; up to 16 pairs travel with the
launch.  The arithmetic of a pixel does not depend on either, so one pair alone (small jobs) and the same
pair in a larger call (large jobs; by table above 16 pairs) must give equal maps, scores and
volumes.  The border recompute is checked through the refinement at odd sizes and widths that leave
half-filled fragments, at the BF16 and FP8 forms' own bars."""
import numpy as np
import pytest
import torch

import oracle
from paper_2305_11566_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,D,W,H", [(3, 1, 64, 40), (3, 33, 301, 130), (7, 16, 256, 128), (9, 48, 1242, 375),
                                     (9, 48, 195, 97), (15, 64, 640, 193), (5, 90, 520, 90), (11, 128, 700, 150)])
def test_small_and_large_jobs_agree(svlib, k, D, W, H):
    ctx = binding.Context(synth.NET_SMALL, k, "fp32")
    try:
        dp = binding.to_device(synth.make_pair(W, H, 4.0 * (D - 1), 300 + W), D)
        one, best, second = ctx.coarse_match([dp], scores=True)
        plain = ctx.coarse_match([dp])
        opts = binding.coarse_opts("zncc", "none")
        vmap, vol = ctx.coarse_match_ex([dp], opts, costs=True)
        for n in (16, 17, 160):
            many, mb, ms = ctx.coarse_match([dp] * n, scores=True)
            mplain = ctx.coarse_match([dp] * n)
            for i in (0, n // 2, n - 1):
                assert torch.equal(many[i], one[0]) and torch.equal(mplain[i], plain[0])
                assert torch.equal(mb[i], best[0]) and torch.equal(ms[i], second[0])
        assert torch.equal(one[0], plain[0])
        n = 160 if W * H < 200000 else 20
        mmap, mvol = ctx.coarse_match_ex([dp] * n, opts, costs=True)
        assert torch.equal(mmap[n - 1], vmap[0]) and torch.equal(mvol[n - 1], vol[0])
    finally:
        ctx.close()


@pytest.mark.parametrize("form,shape", [
    ("bf16", synth.NetShape((16, 48, 32), 16, (80, 16, 48))), ("bf16", synth.NET_SMALL),
    ("fp8", synth.NetShape((32, 64, 32), 96, (32, 64, 48))), ("fp8", synth.NET_WIDE)], ids=["bf16-odd", "bf16", "fp8-odd", "fp8"])
@pytest.mark.parametrize("W,H", [(61, 30), (60, 31), (59, 37), (130, 66), (251, 67)])
def test_border_recompute(svlib, form, shape, W, H):
    k, D = 3, 4
    params = synth.he_normal_weights(shape, 7)
    ctx = binding.Context(shape, k, form)
    try:
        ctx.set_weights(params)
        p = synth.make_pair(W, H, 12.0, 500 + W + H)
        coarse = np.random.default_rng(3).integers(0, D, (H // 4, W // 4)).astype(np.int16)
        Y = ctx.refine([binding.to_device(p, D)], [torch.from_numpy(coarse).cuda()])[0]
        ctx.synchronize()
        if form == "bf16":
            ref = oracle.refine_forward(shape, params, p.left, coarse.astype(np.float64))["Y"]
            top, mean = 0.05, 0.01
        else:
            ref = oracle.refine_forward_q(shape, params, p.left, coarse.astype(np.float64))["Y"]
            top, mean = 0.25, 0.005
        err = np.abs(Y.cpu().numpy().astype(np.float64) - ref)
        assert err.max() <= top and err.mean() <= mean, (err.max(), err.mean())
    finally:
        ctx.close()


@pytest.mark.parametrize("W,H", [(61, 31), (253, 64), (255, 37), (257, 66), (509, 35), (1241, 75)])
@pytest.mark.parametrize("form,shape", [("bf16", synth.NET_SMALL), ("bf16", synth.NET_WIDE), ("fp8", synth.NET_WIDE),
                                        ("bf16", synth.NetShape((16, 32, 16), 16, (32, 32, 32)))],
                         ids=["small", "wide", "fp8", "32-32"])
def test_fused_tail_odd_widths(svlib, form, shape, W, H):
    """The fused decoder tail at odd widths (mixed with an even one) against the separate kernels:
    only BF16 rounding of d3 and of the summed weights lies between them (the forms' bars)."""
    k, D = 3, 4
    ctx = binding.Context(shape, k, form)
    try:
        ctx.set_weights(synth.he_normal_weights(shape, 7))
        sizes = [(W, H), (W + 1, H), (W, H + 1)]
        dps = [binding.to_device(synth.make_pair(w, h, 12.0, 700 + w + h), D) for w, h in sizes]
        rng = np.random.default_rng(5)
        maps = [torch.from_numpy(rng.integers(0, D, (h // 4, w // 4)).astype(np.int16)).cuda() for w, h in sizes]
        fused = ctx.refine(dps, maps)
        ctx.set_option("fused_final", 0)
        apart = ctx.refine(dps, maps)
        ctx.synchronize()
        for (w, h), a, b in zip(sizes, fused, apart):
            d = (a - b).abs()
            assert d.max().item() <= 0.05 and d.mean().item() <= 0.01, (w, h, d.max().item())
            assert d[:, -2:].mean().item() <= 0.01, (w, h)
    finally:
        ctx.close()


@pytest.mark.parametrize("k,D,W,H", [(5, 33, 262, 80), (9, 40, 322, 97), (3, 48, 200, 64), (15, 47, 420, 130)])
def test_half_warp_argmax_ties_and_edges(svlib, k, D, W, H):
    """Disparity ranges of 33-48 run the half-warp layout without scores: textures full of exact
    ties (periods of 3 and 5 quarter-size pixels, flat areas), where the lowest valid disparity must
    win, against the full-warp layout with scores and the exact-integer oracle."""
    rng = np.random.default_rng(k)
    h, w = H // 4, W // 4
    rows = rng.integers(0, 255, (h, 15)).astype(np.uint8)
    left = np.tile(rows[:, :5], (1, w // 5 + 1))[:, :w]
    right = np.tile(rows[:, :3], (1, w // 3 + 1))[:, :w]
    right[: h // 2] = left[: h // 2]
    left[:, w // 2: w // 2 + 20] = 77
    big = [np.zeros((H, W), np.uint8) for _ in range(2)]
    for b, s in zip(big, (left, right)):
        b[: 4 * h, : 4 * w] = np.repeat(np.repeat(s, 4, 0), 4, 1)
    dp = binding.to_device(synth.Pair(big[0], big[1], np.zeros((H, W), np.float32), np.zeros((H, W), bool), 0), D)
    ctx = binding.Context(synth.NET_SMALL, k, "fp32")
    try:
        plain = ctx.coarse_match([dp])[0]
        scored, best, _ = ctx.coarse_match([dp], scores=True)
        many = ctx.coarse_match([dp] * 160)
        assert torch.equal(plain, scored[0]) and torch.equal(plain, many[159])
        want, _, _ = oracle.coarse_match(big[0], big[1], k, D)
        # differences only where FP32 scores cannot tell the oracle's candidates apart
        d = plain.cpu().numpy() != want
        assert d.mean() <= 0.02, d.mean()
    finally:
        ctx.close()
