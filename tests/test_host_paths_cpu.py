"""Host code of the library under conditions a GPU test does not make (tests/hostlib.py)."""
import pytest

import hostlib
from paper_2305_11566_gb300 import binding, synth


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    return hostlib.load(tmp_path_factory.mktemp("host"))


def count(h, name):
    return sum(name in k for k, _ in h.launches())


@pytest.mark.parametrize("failing", ["first allocation", "second allocation", "packing"])
def test_training_after_a_failed_first_call(host, failing):
    """A BF16 context plans its FP32 layers at the first training call.  If one of the plan's allocations
    or the packing of its weights fails, the call fails without a launch, new weights do not touch the
    missing plan, and the next call plans again, with its weights packed before they are used."""
    h = hostlib.Host(host, synth.NET_SMALL, "bf16", [(64, 48)])
    try:
        host.host_clear()
        if failing == "packing":
            host.host_launch_fail_in(1)
        else:
            host.host_fail_in(1 if failing == "first allocation" else 2)
        assert h.train() == (binding.SV_ERR_CUDA if failing == "packing" else binding.SV_ERR_OOM), h.error()
        assert host.host_launches() == 0
        assert h.backward() == binding.SV_ERR_STATE
        w = h.buffer(4 * h.params)
        assert host.sv_set_weights(h.ctx, w, h.params) == binding.SV_OK
        assert count(h, "f32_pack_kernel") == 0
        host.host_clear()
        assert h.train() == binding.SV_OK, h.error()
        names = [k for k, _ in h.launches()]
        pack = [i for i, k in enumerate(names) if "f32_pack_kernel" in k]
        use = [i for i, k in enumerate(names) if "f32_conv_kernel" in k]
        assert len(pack) == 1 and use and pack[0] < use[0]
        assert h.backward() == binding.SV_OK
    finally:
        h.close()


def test_weight_gradient_slots_are_bounded(host):
    """Every pair has weight-gradient slots of its own (19 MB for dec2 of the 32/64/128 net on a 256 x 128
    crop), so a backward of many pairs takes them in ranges: beside the saved activations it needs the
    2 GiB of a group's gradients and 1 GiB of slots at most, 4 % for its tables."""
    h = hostlib.Host(host, synth.NET_WIDE, "fp32", [(256, 128)] * 200, 7, 16)
    try:
        assert h.train() == binding.SV_OK, h.error()
        before = host.host_used()
        host.host_clear()
        assert h.backward() == binding.SV_OK, h.error()
        assert host.host_peak() - before <= 1.04 * (3 << 30), host.host_peak() - before
        # every pair's slots are summed: 200 pairs of 64 tiles in dec2's 128 x 64 grid
        dec2 = [g for k, g in h.launches() if "wgrad_f32_kernel" in k and g[0] % 64 == 0]
        assert sum(g[0] for g in dec2) >= 200 * 64
    finally:
        h.close()
