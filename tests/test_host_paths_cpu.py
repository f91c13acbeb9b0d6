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


def pair_bytes(net, W, H, levels):
    """FP32 bytes of the activations e1 e2 e3 z d1 d2 d3 (those asked for) of one W x H pair."""
    px = [W * H]
    for _ in range(3):
        W, H = (W + 1) // 2, (H + 1) // 2
        px.append(W * H)
    ch = (*net.enc, net.latent, *net.dec)
    at = (1, 2, 3, 3, 2, 1, 0)
    return 4 * sum(px[at[k]] * ch[k] for k in levels)


@pytest.mark.parametrize("room", [1.2, 2.5, 20])
def test_fp32_refine_in_the_memory_that_is_there(host, room):
    """Eight frames refine where the activations of one fit (and none where they do not)."""
    W, H, n = 1242, 375, 8
    h = hostlib.Host(host, synth.NET_WIDE, "fp32", [(W, H)] * n, 9, 48)
    one = pair_bytes(synth.NET_WIDE, W, H, range(7))
    try:
        host.host_limit(host.host_used() + int(0.9 * one))
        assert h.refine() == binding.SV_ERR_OOM and "activations" in h.error()
        host.host_limit(host.host_used() + int(room * one))
        host.host_clear()
        assert h.refine() == binding.SV_OK, h.error()
        assert h.error() == ""
        finals = [g[2] for k, g in h.launches() if "f32_final_kernel" in k]
        assert sum(finals) == n and max(finals) <= room
    finally:
        h.close()


@pytest.mark.parametrize("keep", [False, True])
def test_fp32_training_in_the_memory_that_is_there(host, keep):
    """Four frames train where the decoder activations of all, and the gradients, the encoder's
    activations and the weight-gradient slots of one fit: the encoder is then recomputed.  With room for
    all of them it is not."""
    W, H, n, net = 1242, 375, 4, synth.NET_WIDE
    h = hostlib.Host(host, net, "fp32", [(W, H)] * n, 9, 48)
    try:
        saved = n * pair_bytes(net, W, H, (3, 3, 3, 3, 4, 5, 6))  # z, logvar, eps, mu; d1 .. d3
        enc = pair_bytes(net, W, H, (0, 1, 2))
        slots = 304 * 4 * (9 * 128 * 128 + 128)
        work = pair_bytes(net, W, H, range(7)) + 2 * enc + slots  # one pair's backward
        room = saved + work if not keep else saved + n * (enc + work)
        base = host.host_used()
        host.host_limit(base + room + (8 << 20))
        for _ in range(2):  # the second step finds the first one's workspaces
            host.host_clear()
            assert h.train() == binding.SV_OK, h.error()
            assert h.backward() == binding.SV_OK, h.error()
            names = [k for k, _ in h.launches()]
            enc1 = [g[2] for k, g in h.launches() if "f32_enc1_kernel" in k]
            assert sum(enc1) == (n if keep else 2 * n), enc1
            assert sum("final_dgrad" in k for k in names) == (1 if keep else n)
            assert host.host_peak() <= base + room + (8 << 20)
        h.close()
        h = hostlib.Host(host, net, "fp32", [(W, H)] * n, 9, 48)
        host.host_limit(host.host_used() + saved // 2)
        assert h.train() == binding.SV_ERR_OOM and h.backward() == binding.SV_ERR_STATE
    finally:
        h.close()


def test_bf16_training_gives_scratch_back(host):
    """The scratch and the slots of a backward do not keep a larger training forward from its memory."""
    h = hostlib.Host(host, synth.NET_SMALL, "bf16", [(1242, 375)] * 12, 9, 48)
    try:
        assert h.train() == binding.SV_OK and h.backward() == binding.SV_OK
        for p in h.pairs:
            p.height += 8  # a little more of everything
        host.host_limit(host.host_used())
        assert h.train() == binding.SV_OK, h.error()
    finally:
        h.close()


@pytest.mark.parametrize("form,n", [("fp32", 70000), ("bf16", 30000)])
def test_more_pairs_than_a_grid_is_deep(host, form, n):
    """So many tiny pairs in one call that a launch's grid cannot hold them (FP32), or three saved
    activations of each (BF16), in y or z."""
    h = hostlib.Host(host, synth.NET_SMALL, form, [(12, 12)] * n, 3, 3)
    try:
        for call in (h.refine, h.train, h.loss, h.backward):
            host.host_clear()
            assert call() == binding.SV_OK, (call.__name__, h.error())
            for name in ("f32_final_kernel", "f32_final_ordered", "loss_partial", "final_dgrad"):
                depth = [max(g[1:]) for k, g in h.launches() if name in k]
                assert not depth or sum(depth) == n, (call.__name__, name, depth)
            convert = [g[1] for k, g in h.launches() if "f32_convert" in k]
            assert not convert or sum(convert) == 4 * n  # e3, d1, d2, d3
    finally:
        h.close()


@pytest.mark.parametrize("form", ["fp32", "bf16", "table1"])
def test_captured_tables_outlive_their_call(host, form):
    """Copies recorded in a caller's stream capture read, at replay, what they read at capture; the
    memory is the graph's."""
    t1 = form == "table1"
    h = hostlib.Host(host, form if t1 else synth.NET_SMALL, "fp32" if t1 else form, [(64, 48), (40, 36)])
    calls = ([h.refine] if form != "bf16" else []) + [h.train] + ([] if t1 else [h.loss, h.backward])
    try:
        for call in calls:
            assert call() == binding.SV_OK, h.error()
        host.host_clear()
        host.host_capture(1)
        for call in calls:
            assert call() == binding.SV_OK, h.error()
        host.host_capture(0)
        assert host.host_copies() >= len(calls)
        assert host.host_stale_copies() == 0
        assert host.host_drop_graph() == host.host_copies()
        for call in calls:  # nothing is kept for a call that is not captured
            assert call() == binding.SV_OK, h.error()
        assert host.host_drop_graph() == 0
    finally:
        host.host_capture(0)
        h.close()


@pytest.mark.parametrize("form", ["bf16", "fp8"])
def test_networks_too_wide_for_the_tensor_core_form(host, form):
    """Widths whose staged rows alone exceed shared memory are refused when the context is created (planning
    them had no end); FP32 takes them."""
    wide = synth.NetShape((256, 256, 256), 256, (256, 256, 256))
    ctx = hostlib.ctypes.c_void_p()
    cfg = binding.make_config(wide, 9, form)
    assert host.sv_create(hostlib.ctypes.byref(cfg), 0, hostlib.ctypes.byref(ctx)) == binding.SV_ERR_UNSUPPORTED
    assert not ctx.value
    h = hostlib.Host(host, wide, "fp32", [(64, 48)])
    try:
        assert h.refine() == binding.SV_OK, h.error()
    finally:
        h.close()
