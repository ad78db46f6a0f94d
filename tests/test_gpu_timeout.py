"""A bounded device-side wait that runs out is reported, not hung on, and leaves the context usable.

The only form in which this is run on a GPU: rrm_options.wait_limit = 0 on the three tensor-core kernels.  There
every role of a thread block (copy producers, filter loader, MMA issuer, epilogue) meets its first wait BEFORE it
has issued any asynchronous copy or MMA, so a wait that gives up at once lets the block leave with nothing in
flight: it frees its tensor memory and returns.  The host then reads bit 1 of rrm_stats.error_word and gets
RRM_ERR_TIMEOUT from rrm_get_stats.  After the limit is restored and the errors are cleared, a keyframe rebuilds
the state and the next frames match the CPU oracle again."""
import numpy as np
import pytest
import torch

import workloads as wl
from workloads.nets import LayerSpec
from oracle import rrm_oracle as orc
from helpers import dev, pack_bits_nhwc

pytestmark = pytest.mark.gpu

TIMEOUT_STATUS, TIMEOUT_BIT = -6, 2


def test_options_round_trip_and_validation():
    import paper_1802_09723_b200 as rrm
    layer = rrm.layer_from_spec(wl.fc6_i8(c_in=256, c_out=128)[0])
    o = layer.options()
    assert o["wait_limit"] == 1 << 20 and abs(o["stack_dense_activity"] - 0.75) < 1e-6 and o["stack_reprobe"] == 15
    assert o["layer_dense_activity"] > 1.0 and o["layer_delta_activity"] > 1.0            # the per-layer choice is opt-in
    layer.set_options(wait_limit=123, fc_dense_rows=0.5)
    o2 = layer.options()
    assert o2["wait_limit"] == 123 and abs(o2["fc_dense_rows"] - 0.5) < 1e-6 and o2["stack_reprobe"] == 15
    with pytest.raises(rrm.RRMError):
        layer.set_options(stack_reprobe=0)
    with pytest.raises(rrm.RRMError):
        layer.set_options(layer_dense_activity=0.2, layer_delta_activity=0.5)
    layer.close()


def test_few_row_fc_kernel_reports_a_wait_that_ran_out_and_recovers():
    import paper_1802_09723_b200 as rrm
    c_in, c_out, T = 1024, 512, 4
    spec = wl.fc6_i8(c_in=c_in, c_out=c_out)[0]
    seq = wl.fc_run_sequence(frames=T + 2, c_in=c_in, rho=0.05, seed=5)
    layer = rrm.layer_from_spec(spec)
    frames = dev(seq)
    Y = layer.new_output(frames=T)
    layer.dense_seq(frames[:T], Y, T)                         # healthy run first: the tensor-core kernel is the one in use
    for t in range(T):
        np.testing.assert_array_equal(Y[t].cpu().numpy().astype(np.int64), orc.dense_forward([spec], seq[t])[0][1])
    assert layer.stats(0)["error_word"] == 0
    layer.set_options(wait_limit=0)
    layer.dense_seq(frames[:T], Y, T)
    st = layer.stats(0, check=False)
    assert st["status"] == TIMEOUT_STATUS and st["error_word"] & TIMEOUT_BIT, st
    with pytest.raises(rrm.RRMError):
        layer.stats(0)
    # the context is intact: restore the limit, clear the flag, rebuild the state, step on
    layer.set_options(wait_limit=1 << 20)
    layer.clear_errors()
    layer.keyframe(frames[0], None)
    Y1 = layer.new_output()
    for t in range(1, T + 2):
        layer.step(frames[t], Y1)
        np.testing.assert_array_equal(Y1.cpu().numpy().astype(np.int64), orc.dense_forward([spec], seq[t])[0][1])
    assert layer.stats(0)["error_word"] == 0
    layer.close()


def test_tensor_core_conv_reports_a_wait_that_ran_out_and_recovers():
    import paper_1802_09723_b200 as rrm
    specs = wl.alexnet_convs("i8", hw=99, scale=8)
    video = wl.moving_rect_video(frames=4, hw=99, dtype="i8", seed=9, side=(12, 24))
    net = rrm.net_from_specs(specs, variant="tensor")
    out = net.new_output()
    net.step(dev(video[0]), out)
    assert net.stats(0)["error_word"] == 0 and net.stats(0)["variant"] == 2       # the tensor-core kernel runs these layers
    net.set_options(wait_limit=0)
    net.step(dev(video[1]), out)                               # the first layer's thread blocks give up at their first wait
    st = net.stats(0, check=False)
    assert st["status"] == TIMEOUT_STATUS and st["error_word"] & TIMEOUT_BIT, st
    net.set_options(wait_limit=1 << 20)
    net.clear_errors()
    net.keyframe(dev(video[1]), out)                           # a precise inference replaces the inconsistent state
    for t in (2, 3):
        net.step(dev(video[t]), out)
        _, P = orc.dense_forward(specs, video[t])
        for l in range(len(specs)):
            np.testing.assert_array_equal(net.projection(l).cpu().numpy().astype(np.int64), P[l])
    assert net.stats(0)["error_word"] == 0
    net.close()


def _lone_layer(dtype, hw):
    rng = np.random.default_rng(hw[1])
    sp = LayerSpec("conv", dtype, 40, hw[0], hw[1], 36, 3, 3, 1, 1, src=0, act="sign" if dtype == "bin" else "none", theta=1)
    sp.weight = ((rng.integers(0, 2, size=(36, 40, 3, 3)) * 2 - 1).astype(np.int8) if dtype == "bin" else
                 rng.integers(-127, 128, size=(36, 40, 3, 3)).astype(np.int8))
    sp.bias = rng.integers(-500, 501, size=36).astype(np.int32)
    video = rng.integers(0, 2, size=(4, 1, 40) + hw) * 2 - 1 if dtype == "bin" else rng.integers(0, 128, size=(4, 1, 40) + hw)
    return [sp], video.astype(np.int8)


@pytest.mark.parametrize("dtype,kernel", [("f32", "windows"), ("bin", "windows"), ("i8", "rows"), ("bin", "rows")])
def test_every_tensor_core_conv_kernel_reports_a_wait_that_ran_out_and_recovers(dtype, kernel):
    """windows: the kernel that keeps windows of the input in shared memory; rows: the one that gathers compacted rows, which
    takes what is too wide for such a window."""
    import paper_1802_09723_b200 as rrm
    if kernel == "rows":
        specs, video = _lone_layer(dtype, (3, 900))
    elif dtype == "bin":
        specs, video = _lone_layer(dtype, (20, 21))
    else:
        specs = wl.alexnet_convs(dtype, hw=99, scale=8)
        video = wl.moving_rect_video(frames=4, hw=99, dtype=dtype, seed=9, side=(12, 24))
    frames = [dev(pack_bits_nhwc(f).view(np.int32)) if dtype == "bin" else dev(f) for f in video]
    net = rrm.net_from_specs(specs, variant="tensor")
    out = net.new_output()
    net.step(frames[0], out)
    assert net.stats(0)["error_word"] == 0 and net.stats(0)["variant"] == 2       # a tensor-core kernel runs these layers
    net.set_options(wait_limit=0)
    net.step(frames[1], out)                                   # the first layer's thread blocks give up at their first wait
    st = net.stats(0, check=False)
    assert st["status"] == TIMEOUT_STATUS and st["error_word"] & TIMEOUT_BIT, st
    net.set_options(wait_limit=1 << 20)
    net.clear_errors()
    net.keyframe(frames[1], out)                               # a precise inference replaces the inconsistent state
    for t in (2, 3):
        net.step(frames[t], out)
        _, P = orc.dense_forward(specs, video[t])
        for l in range(len(specs)):
            got = net.projection(l).cpu().numpy()
            if dtype == "f32":
                assert float(np.abs(got - P[l]).max()) <= 1e-4 * float(np.abs(P[l]).max())
            else:
                np.testing.assert_array_equal(got.astype(np.int64), P[l])
    assert net.stats(0)["error_word"] == 0
    net.close()
