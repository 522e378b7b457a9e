"""Which kernels the library's host code launches, and where: run over a stand-in CUDA runtime
(fake_runtime.py) that enforces the launch rules of each device.  CPU only."""
import ctypes

import numpy as np
import pytest

import fake_runtime
import paper_2607_01735_gb300 as rb
from fake_runtime import Context, launches


@pytest.fixture(scope="module")
def loaded():
    return fake_runtime.load()


@pytest.fixture
def lib(loaded):
    loaded.fake_reset()
    yield loaded
    loaded.fake_reset()


# ------------------------------------------------------------------ a second device
@pytest.mark.parametrize("n,opts", [(1023, {}), (1368, {}), (1023, {"fma": 1}), (1500, {"fma": 1}), (4095, {}),
                                    (900, {"kernel": rb.RBGS_KERNEL_WAVEFRONT})])
def test_sweeps_run_on_a_second_device(lib, n, opts):
    """A kernel's raised shared-memory limit belongs to the device it was raised on."""
    for device in (0, 1):
        lib.fake_set_device(device)
        c = Context(lib, n, **opts)
        st, calls = c.sweep(40)
        assert st == 0, lib.rbgs_last_error()
        assert calls and all(d == device for kind, _, _, d in calls if kind != "graph")
        c.close()


@pytest.mark.parametrize("n,opts", [(127, {}), (1023, {}), (1023, {"fma": 1}), (1500, {"fma": 1})])
def test_sweeps_run_after_a_device_reset(lib, n, opts):
    lib.fake_set_device(4)  # used by no other test, whose kernels keep their raised limits
    for _ in range(2):
        c = Context(lib, n, **opts)
        st, calls = c.sweep(40)
        assert st == 0 and calls, lib.rbgs_last_error()
        assert n > 1368 or _kinds(calls) <= {"cooperative", "plain"} and any("resident" in k for _, k, _, _ in calls)
        c.close()
        lib.fake_device_reset()


def test_refined_solve_runs_on_a_second_device(lib):
    for device in (0, 1):
        lib.fake_set_device(device)
        c = Context(lib, 900, precision=rb.RBGS_FP32_REFINE, max_sweeps=200, inner_sweeps=100)
        lib.fake_clear_log()
        assert lib.rbgs_solve(c.ctx, 0.0, None, None) == rb.RBGS_ENOTCONV, lib.rbgs_last_error()
        inner = [kind for kind, name, _, _ in launches(lib) if "resident" in name]
        assert inner == ["cooperative"] * 2
        c.close()


def test_cooperative_launches_fit_a_smaller_second_device(lib):
    lib.fake_set_sms(2, 60)  # a device that no other test uses: its SM count is asked for once
    for n, opts in ((511, {}), (511, {"fma": 1}), (4095, {})):
        for device, sms in ((0, 152), (2, 60)):
            lib.fake_set_device(device)
            c = Context(lib, n, **opts)
            st, calls = c.sweep(40)
            assert st == 0, lib.rbgs_last_error()
            blocks = [b for kind, name, b, _ in calls if kind == "cooperative"]
            assert blocks and (n > 2048 or max(blocks) <= sms)
            c.close()


@pytest.mark.parametrize("Cin,Cout", [(32, 32), (128, 128), (192, 64)])
def test_convolutions_run_on_a_second_device(lib, Cin, Cout):
    B, H, W = 2, 66, 66
    aligned = lambda n: (lambda a: a[(-a.ctypes.data % 16) // a.itemsize:])(np.zeros(n + 64, np.uint16))
    x, w, g, t = (aligned(k) for k in (B * H * W * Cin, 9 * Cin * Cout, B * H * W * Cout, 9 * Cin * Cout))
    y, dx, dw = (np.zeros(k, np.float32) for k in (B * H * W * Cout, B * H * W * Cin, 9 * Cin * Cout))
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    lib.rbgs_conv_set_engine(2)  # gathers: tensor maps need a driver
    try:
        for device in (0, 1):
            lib.fake_set_device(device)
            for engine in (2, 0):
                lib.rbgs_conv_set_engine(engine)
                assert lib.rbgs_conv_forward(p(x), p(w), None, p(y), B, H, W, Cin, Cout, 3, 0, 1, None) == 0
            lib.rbgs_conv_set_engine(2)
            for kind in (1, 2, 3):
                lib.rbgs_conv_set_wgrad_kernel(kind)
                assert lib.rbgs_conv_backward(p(x), p(w), p(g), p(dx), p(dw), None, p(t), B, H, W, Cin, Cout, 3, 0,
                                              None) == 0, lib.rbgs_last_error()
    finally:
        lib.rbgs_conv_set_wgrad_kernel(0)
        lib.rbgs_conv_set_engine(0)


# ------------------------------------------------------------------ refused cooperative launches
def _kinds(calls):
    return {kind for kind, *_ in calls}


@pytest.mark.parametrize("n,opts", [(31, {}), (255, {}), (255, {"fma": 1}), (900, {"fma": 1})])
def test_sweeps_go_on_when_the_cooperative_launch_is_refused(lib, n, opts):
    """A process that may use only part of the SMs has cooperative launches refused: the sweeps
    then run one launch per colour, and later calls do not try again."""
    c = Context(lib, n, **opts)
    lib.fake_cooperative(1, 1)
    for k in (40, 2, 40):
        st, calls = c.sweep(k)
        assert st == 0, lib.rbgs_last_error()
        assert calls and _kinds(calls) <= {"plain", "graph"}
        assert not any("resident" in name for _, name, _, _ in calls)
    lib.fake_cooperative(1, 0)
    st, calls = c.sweep(40)
    assert st == 0 and _kinds(calls) <= {"plain", "graph"}
    c.close()


def test_refinement_goes_on_when_the_cooperative_launch_is_refused(lib):
    for n in (127, 511):
        c = Context(lib, n, precision=rb.RBGS_FP32_REFINE, max_sweeps=200, inner_sweeps=100)
        lib.fake_cooperative(1, 1)
        lib.fake_clear_log()
        assert lib.rbgs_solve(c.ctx, 0.0, None, None) == rb.RBGS_ENOTCONV, lib.rbgs_last_error()
        assert "cooperative" not in _kinds(launches(lib))
        lib.fake_cooperative(1, 0)
        c.close()


def test_device_without_cooperative_launches(lib):
    """The attribute is asked for once per device: this one is used by no other test."""
    lib.fake_set_device(3)
    lib.fake_cooperative(0, 0)
    for opts in ({}, {"fma": 1}):
        c = Context(lib, 255, **opts)
        st, calls = c.sweep(40)
        assert st == 0 and calls and _kinds(calls) <= {"plain", "graph"}
        c.close()


# ------------------------------------------------------------------ several solvers at once
def _tiles(calls):
    return [blocks for kind, name, blocks, _ in calls if kind == "cooperative" and "resident" in name]


@pytest.mark.parametrize("n,opts", [(127, {}), (255, {"fma": 1})])
def test_solvers_on_several_streams_share_the_device(lib, n, opts):
    """A launch takes the whole device alone, and a part of it while other streams are busy (here:
    with a second's worth of sweeps each); contexts of one stream or of another device do not count."""
    lone = Context(lib, n, stream=101, **opts)
    whole = _tiles(lone.sweep(20)[1])
    assert whole and whole[0] > 76
    lone.close()
    busy = [Context(lib, n, stream=201 + q, **opts) for q in range(7)]
    parts = [_tiles(c.sweep(1000000)[1])[0] for c in busy]
    assert parts[0] == whole[0] and all(p <= 152 // 2 for p in parts[1:]) and parts[-1] <= 152 // 6
    same = Context(lib, n, stream=201, **opts)
    assert _tiles(same.sweep(20)[1])[0] <= 152 // 6  # six other streams besides its own
    lib.fake_set_device(1)
    other = Context(lib, n, stream=301, **opts)
    assert _tiles(other.sweep(20)[1]) == whole
    other.close()
    lib.fake_set_device(0)
    for c in busy:
        c.close()  # waits for its stream
    got = [_tiles(same.sweep(20)[1]) for _ in range(3)]
    assert got[-1] == whole  # the third launch in a row with no other stream busy
    same.close()


def test_captured_launches_neither_share_nor_count(lib):
    lib.fake_capture.argtypes = [ctypes.c_void_p]
    lib.fake_set_device(5)
    busy, caught, later = (Context(lib, 127, stream=q) for q in (401, 402, 403))
    lib.fake_capture(402)
    assert _tiles(caught.sweep(1000000)[1])[0] == 152
    lib.fake_capture(2 ** 64 - 1)
    assert _tiles(busy.sweep(1000000)[1])[0] == 152  # the captured launch is not at work
    lib.fake_capture(402)
    assert _tiles(caught.sweep(1000000)[1])[0] == 152  # and takes the plan it would take alone
    lib.fake_capture(2 ** 64 - 1)
    assert _tiles(later.sweep(20)[1])[0] <= 76
    for c in (busy, caught, later):
        c.close()


def test_any_sweep_count_leaves_the_clock_in_range(lib):
    lib.fake_set_device(5)
    a, b = Context(lib, 127, stream=501), Context(lib, 127, stream=502)
    for k in (2 ** 62, 2 ** 62, 5):
        assert a.sweep(k)[0] == 0
    assert _tiles(b.sweep(20)[1])[0] <= 76  # still counted as busy
    a.close()
    b.close()


# ------------------------------------------------------------------ single sweeps
@pytest.mark.parametrize("n,kernels", [(255, ["half_sweep"] * 2), (511, ["persistent_sweeps"]),
                                       (1023, ["persistent_sweeps"]), (4095, ["persistent_sweeps"])])
def test_a_single_sweep_takes_the_fewest_launches(lib, n, kernels):
    """One sweep of a grid that several sweeps would run in tiles: the grid-barrier launch from
    416^2 on, one launch per colour below."""
    c = Context(lib, n)
    st, calls = c.sweep(1)
    assert st == 0 and len(calls) == len(kernels)
    assert all(want in name for want, (_, name, _, _) in zip(kernels, calls)), calls
    c.close()


# ------------------------------------------------------------------ the automatic choice's limits
@pytest.mark.parametrize("n,opts,kernel", [
    (1368, {}, "resident"), (1369, {}, "persistent"), (1368, {"fma": 1}, "resident"), (1369, {"fma": 1}, "wavefront"),
    (3000, {"fma": 1}, "wavefront"), (63, {"fma": 1}, "resident"),
    (1400, {"fma": 1, "kernel": rb.RBGS_KERNEL_COLOUR}, "fused_half_sweep"), (415, {}, "resident")])
def test_automatic_choice_of_the_sweeps(lib, n, opts, kernel):
    c = Context(lib, n, **opts)
    st, calls = c.sweep(9)
    names = [name for _, name, _, _ in calls if not any(w in name for w in ("absmax", "prepare"))]
    assert st == 0 and names and all(kernel in name for name in names), names
    c.close()


@pytest.mark.parametrize("n,kernel", [(127, "resident"), (1000, "resident"), (1001, "wavefront"), (4095, "wavefront")])
def test_automatic_choice_of_the_inner_sweeps(lib, n, kernel):
    c = Context(lib, n, precision=rb.RBGS_FP32_REFINE, max_sweeps=100, inner_sweeps=100)
    lib.fake_clear_log()
    assert lib.rbgs_solve(c.ctx, 0.0, None, None) == rb.RBGS_ENOTCONV
    assert any(kernel in name for _, name, _, _ in launches(lib))
    assert not any(k in name for _, name, _, _ in launches(lib) for k in {"resident", "wavefront"} - {kernel})
    c.close()


# ------------------------------------------------------------------ the network's buffers
def test_network_buffers_are_what_a_pass_needs(lib):
    """A forward pass holds the activations and its output; a training step adds the FP32 gradients
    of the concatenations and pooled tensors and two bf16 ones, the mma.sync engine one more FP32."""
    B, H = 2, 64
    P = B * H * H
    x, y, m = np.zeros((P, 4), np.float32), np.zeros(P, np.float32), np.ones(P, np.float32)
    p = lambda a: ctypes.c_void_p(a.ctypes.data)
    net = ctypes.c_void_p()
    lib.rbgs_unet_create.argtypes = [ctypes.c_uint64, ctypes.c_void_p, ctypes.POINTER(ctypes.c_void_p)]
    lib.rbgs_unet_train_step.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_int] * 3 + [ctypes.c_float] + [ctypes.c_void_p] * 2
    lib.rbgs_unet_destroy.restype = None
    before = lib.fake_memory_in_use()
    assert lib.rbgs_unet_create(1, None, ctypes.byref(net)) == 0
    weights = lib.fake_memory_in_use()
    channels = 16 + 32 + 32 + 96 + 32 + 32 + (32 + 64 + 64 + 192 + 64 + 64) / 4 + (64 + 128 + 128 + 384 + 128 + 128) / 16 \
        + (128 + 256 + 256) / 64
    acts = int(P * channels * 2) + P * 8 * 4 + 8
    lib.rbgs_conv_set_engine(2)  # gathers: tensor maps need a driver
    try:
        assert lib.rbgs_unet_forward(net, p(x), p(y), B, H, H) == 0
        assert lib.fake_memory_in_use() - weights == acts
        step = lambda: lib.rbgs_unet_train_step(net, p(x), p(y), p(m), B, H, H, 1e-3, None, None)
        summed = 96 + 192 / 4 + 384 / 16 + 32 / 4 + 64 / 16 + 128 / 64
        for _ in range(2):
            assert step() == 0, lib.rbgs_last_error()
            assert lib.fake_memory_in_use() - weights == acts + int(P * summed * 4) + 2 * P * 32 * 2
        lib.rbgs_conv_set_engine(1)
        assert step() == 0, lib.rbgs_last_error()
        assert lib.fake_memory_in_use() - weights == acts + int(P * summed * 4) + 2 * P * 32 * 2 + P * 32 * 4
        assert lib.rbgs_unet_forward(net, p(x), p(y), 1, H, H) == 0  # another size frees them
        assert lib.fake_memory_in_use() - weights <= acts
        # out of memory part way: nothing is kept, and a smaller size still works
        lib.fake_memory_limit(lib.fake_memory_in_use() + acts)
        assert lib.rbgs_unet_train_step(net, p(x), p(y), p(m), B, H, H, 1e-3, None, None) == 2
        assert lib.fake_memory_in_use() == weights
        assert lib.rbgs_unet_forward(net, p(x), p(y), 1, H, H) == 0
    finally:
        lib.rbgs_conv_set_engine(0)
        lib.fake_memory_limit(2 ** 63)
        lib.rbgs_unet_destroy(net)
    assert lib.fake_memory_in_use() == before
