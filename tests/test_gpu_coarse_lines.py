"""Path and filter kernels of the coarse-stage variants at the disparity ranges where their lane
layouts change, line counts that do not fill a warp, volumes at 4-byte alignment and batches of
several parts.  Census costs with integer penalties are exact in FP32, so volumes and maps are compared
bit for bit with the oracle; parts and alignment with the same pair alone."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
from paper_2305_11566_gb300 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(svlib):
    c = binding.Context(synth.NET_SMALL, 3, "fp32")
    yield c
    c.close()


@pytest.mark.parametrize("D,W,H", [(1, 20, 12), (2, 33, 17), (8, 64, 32), (9, 71, 45), (16, 130, 29), (17, 69, 60),
                                   (32, 140, 52), (33, 133, 36), (48, 262, 41), (49, 260, 33), (64, 300, 44),
                                   (65, 261, 28), (96, 400, 24), (97, 388, 36), (128, 516, 32)])
@pytest.mark.parametrize("npaths", [1, 2, 3, 4])
def test_sgm_layouts_bit_exact(ctx, D, W, H, npaths):
    p = synth.make_pair(W, H, 4.0 * D, 40 + W + D)
    C = oracle.census_volume(oracle.downsample4(p.left), oracle.downsample4(p.right), 5, D)
    A = oracle.sgm(C, 2.0, 12.0, npaths)
    dp = binding.to_device(p, D)
    o = binding.coarse_opts("census", "sgm", census_window=5, P1=2.0, P2=12.0, npaths=npaths)
    disp, vols = ctx.coarse_match_ex([dp], o, costs=True)
    assert np.array_equal(vols[0].cpu().numpy(), A)
    assert np.array_equal(disp[0].cpu().numpy(), oracle.sgm_wta(A))
    assert torch.equal(ctx.coarse_match_ex([dp], o)[0], disp[0])
    # the caller's volume at 4-byte alignment
    h, w = dp.coarse_hw
    buf = torch.zeros(h * w * D + 1, dtype=torch.float32, device="cuda")
    d2 = torch.empty_like(disp[0])
    s = binding.lib().sv_coarse_match_ex(ctx.handle, binding._pairs_array([dp]), 1, ctypes.byref(o), binding._ptrs([d2]),
                                         binding._ptrs([buf[1:]]), binding._stream(None))
    assert s == binding.SV_OK
    assert torch.equal(buf[1:].view(h, w, D), vols[0]) and torch.equal(d2, disp[0]) and buf[0].item() == 0.0


@pytest.mark.parametrize("D,W,H", [(1, 20, 12), (7, 41, 40), (16, 72, 36), (48, 260, 70), (65, 301, 26)])
def test_dt_lines(ctx, D, W, H):
    p = synth.make_pair(W, H, 4.0 * D, 60 + W)
    C = oracle.census_volume(oracle.downsample4(p.left), oracle.downsample4(p.right), 3, D)
    A = oracle.dt_aggregate(C, oracle.downsample4(p.left), 6.0, 25.0, 3)
    o = binding.coarse_opts("census", "dt", census_window=3, dt_sigma_s=6.0, dt_sigma_r=25.0, dt_iters=3)
    _, vols = ctx.coarse_match_ex([binding.to_device(p, D)], o, costs=True)
    np.testing.assert_allclose(vols[0].cpu().numpy(), A, rtol=0, atol=2e-3)  # census + DT bar of the variants


@pytest.mark.parametrize("cost,agg", [("zncc", "sgm"), ("census", "dt"), ("zncc", "none"), ("census", "none")])
def test_parts_equal_single_calls(ctx, cost, agg):
    """Batches whose volumes need several parts, of mixed sizes: every pair as if alone."""
    specs = [(1242, 375, 48), (640, 193, 25), (1242, 375, 48), (322, 97, 13)]
    dps = [binding.to_device(synth.make_pair(W, H, 4.0 * D, 80 + i), D) for i, (W, H, D) in enumerate(specs)]
    o = binding.coarse_opts(cost, agg, P1=0.1, P2=0.5, smp=True, median=True)
    alone = [ctx.coarse_match_ex([dp], o)[0] for dp in dps]
    many = ctx.coarse_match_ex(dps * 60, o)
    for i, m in enumerate(many):
        assert torch.equal(m, alone[i % 4]), i
