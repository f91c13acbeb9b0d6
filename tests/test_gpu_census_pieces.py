"""Census costs of calls with few rows, whose rows are cut into pieces of 32 to 2048 pixels: widths around
the pieces' ends, disparity ranges that reach one or more pieces back, mixed sizes.  Bit-exact."""
import numpy as np
import pytest

import oracle
from paper_2305_11566_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def want(p, D, kc=5):
    return oracle.census_volume(oracle.downsample4(p.left), oracle.downsample4(p.right), kc, D)


@pytest.mark.parametrize("sizes", [
    [(4 * 31, 12, 9)], [(4 * 32, 12, 32)], [(4 * 33 + 1, 13, 33)], [(4 * 64, 40, 5)], [(4 * 65 + 3, 12, 65)],
    [(4 * 129, 16, 128)], [(4 * 700, 12, 100)], [(640, 128, 48)], [(4 * 200, 400, 20)],
    [(4 * 2049, 12, 17)] + [(4 * 31, 400, 1)] * 7,
    [(4 * 300 + 2, 24, 77), (4 * 31, 60, 1), (4 * 97, 12, 97)],
])
def test_census_volume_bit_exact(svlib, sizes):
    ctx = binding.Context(synth.NET_SMALL, 3, "fp32")
    try:
        pairs = [synth.make_pair(W, H, 3.0 * D, 900 + W) for W, H, D in sizes]
        dps = [binding.to_device(p, D) for p, (_, _, D) in zip(pairs, sizes)]
        disp, vols = ctx.coarse_match_ex(dps, binding.coarse_opts("census", census_window=5), costs=True)
        for p, (_, _, D), d, v in zip(pairs, sizes, disp, vols):
            C = want(p, D)
            assert np.array_equal(v.cpu().numpy(), C)
            assert np.array_equal(d.cpu().numpy(), oracle.sgm_wta(C))
    finally:
        ctx.close()
