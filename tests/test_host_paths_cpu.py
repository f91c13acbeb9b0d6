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
