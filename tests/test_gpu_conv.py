"""GPU parity of the convolution path (single layers and layer stacks) against the CPU oracle.
Integer and binary layers must match bit for bit; fp32 layers within 1e-4 * max|P_dense| per
frame (the accumulated projection is compared at every frame, so drift would show)."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import workloads as wl
from workloads.nets import LayerSpec, out_hw
from oracle import rrm_oracle as orc
from helpers import dev, pack_bits_nhwc, unpack_bits_nhwc

pytestmark = pytest.mark.gpu
F32_TOL = 1e-4


def _rrm():
    import paper_1802_09723_b200 as rrm
    return rrm


def _frame_to_dev(specs, frame):
    if specs[0].dtype == "bin":
        return dev(pack_bits_nhwc(frame).view(np.int32))
    return dev(frame)


def _out_kind(s):
    if s.dtype == "f32":
        return "f32"
    if s.act == "sign":
        return "bin"
    return "i8" if s.shift >= 0 else "i32"


def _compare(specs, net, frame, t, check_tensors=True):
    tens_d, P_d = orc.dense_forward(specs, frame)
    for l, s in enumerate(specs):
        P = net.projection(l).cpu().numpy()
        if s.dtype == "f32":
            scale = float(np.abs(P_d[l]).max())
            err = float(np.abs(P.astype(np.float64) - P_d[l]).max())
            assert err <= F32_TOL * scale, f"frame {t} layer {l} ({s.name}): err {err:.3e} scale {scale:.3e}"
        else:
            np.testing.assert_array_equal(P.astype(np.int64), P_d[l], err_msg=f"frame {t} layer {l} ({s.name})")
        if not check_tensors:
            continue
        T = net.tensor(l + 1).cpu().numpy()
        kind = _out_kind(s)
        if kind == "bin":
            np.testing.assert_array_equal(unpack_bits_nhwc(T.view(np.uint32), s.c_out), tens_d[l + 1],
                                          err_msg=f"frame {t} tensor {l + 1}")
        elif kind == "f32":
            scale = max(1e-30, float(np.abs(tens_d[l + 1]).max()))
            assert float(np.abs(T - tens_d[l + 1]).max()) <= F32_TOL * max(scale, float(np.abs(P_d[l]).max()))
        else:
            np.testing.assert_array_equal(T.astype(np.int64), tens_d[l + 1], err_msg=f"frame {t} tensor {l + 1}")


def _run(specs, video, n=1, check_frames=None, stats=False, keyframe_at=(), variant="auto", stats_frames=()):
    """stats: compare every frame's counters with the literal recurrence (small stacks).  stats_frames: the same at
    the named frames only, the recurrence being brought to the frame before by a dense pass (full-size stacks)."""
    rrm = _rrm()
    net = rrm.net_from_specs(specs, n=n, variant=variant)
    out = net.new_output()
    rec = orc.Recurrence(specs, n=n) if stats else None
    if rec is not None:
        # a fresh library state is the stack's response to the all-zero input pattern (all -1 for a
        # binary input); bring the literal recurrence to the same state
        rec.step(np.full_like(video[0], -1 if specs[0].dtype == "bin" else 0))
    for t in range(video.shape[0]):
        x = _frame_to_dev(specs, video[t])
        if t in keyframe_at:
            net.keyframe(x, out)
        else:
            net.step(x, out)
        if rec is not None:
            rec.step(video[t])
            if t not in keyframe_at:
                for l in range(len(specs)):
                    st = net.stats(l)
                    assert st["error_word"] == 0
                    if specs[0].dtype != "f32" or l == 0:
                        assert st["nnz_elems"] == rec.nnz[l], (t, l, st, rec.nnz[l])
                        assert st["active_macs"] == rec.macs[l], (t, l, st, rec.macs[l])
        if t in stats_frames:
            one = orc.Recurrence(specs, n=n)
            one.reset_to(video[t - 1])
            one.step(video[t])
            for l in range(len(specs)):
                st = net.stats(l)
                assert st["error_word"] == 0 and st["nnz_elems"] != -1, (t, l, st)
                assert st["dense_macs"] == orc.layer_macs(specs[l]) * n
                if specs[0].dtype != "f32" or l == 0:
                    assert st["nnz_elems"] == one.nnz[l], (t, l, st, one.nnz[l])
                    assert st["active_macs"] == one.macs[l], (t, l, st, one.macs[l])
                assert 0 < st["active_out_pixels"] <= st["out_pixels"] and st["nnz_elems"] <= st["in_elems"]
        if check_frames is None or t in check_frames:
            _compare(specs, net, video[t], t)
            # the caller-owned output equals the last tensor
            last = net.tensor(len(specs))
            assert torch.equal(out, last)
    net.close()


# ------------------------------------------------------------------ config 1
def test_cfg1_single_conv_fp32_all_frames():
    specs = wl.single_conv_f32()
    video = wl.block_redraw_sequence()
    _run(specs, video, stats=True)


def _spec(dtype, c_in, hw, c_out, k, s, p, rng, **kw):
    sp = LayerSpec("conv", dtype, c_in, hw[0], hw[1], c_out, k, k, s, p, src=0, **kw)
    if dtype == "f32":
        sp.weight = rng.standard_normal((c_out, c_in, k, k)).astype(np.float32) * np.float32(0.1)
        sp.bias = rng.standard_normal(c_out).astype(np.float32)
    elif dtype == "i8":
        sp.weight = rng.integers(-127, 128, size=(c_out, c_in, k, k)).astype(np.int8)
        sp.bias = rng.integers(-500, 501, size=c_out).astype(np.int32)
    else:
        sp.weight = (rng.integers(0, 2, size=(c_out, c_in, k, k)) * 2 - 1).astype(np.int8)
        sp.bias = rng.integers(-5, 6, size=c_out).astype(np.int32)
    return sp


def _video(dtype, c, hw, frames, n, rng):
    kind = {"f32": "f32_relu", "i8": "i8", "bin": "pm1"}[dtype]
    h, w = hw
    seq = wl.block_redraw_sequence(frames=frames, c=c, hw=max(h, w), frac=0.08, block=3, dtype=kind,
                                   seed=int(rng.integers(1, 1 << 30)), n=n)[:, :, :, :h, :w].copy()
    seq[2] = seq[1]                                  # zero delta
    if dtype == "bin":
        seq[3] = -seq[2]                             # every element changes
    elif dtype == "i8":
        seq[3] = 127 - seq[2]
    else:
        seq[3] = seq[2] + np.float32(0.5)
    return seq


@pytest.mark.parametrize("dtype", ["f32", "i8", "bin"])
@pytest.mark.parametrize("c_in,c_out,hw,k,s,p", [
    (3, 5, (9, 11), 3, 1, 1), (16, 70, (13, 13), 3, 1, 1), (8, 12, (17, 15), 5, 2, 2), (5, 9, (12, 12), 1, 1, 0),
    (4, 8, (20, 19), 1, 2, 0), (3, 6, (35, 35), 11, 4, 0), (3, 8, (30, 30), 7, 2, 3), (40, 33, (7, 7), 3, 1, 0),
    (64, 16, (10, 10), 3, 1, 1)])
def test_single_layer_shapes(dtype, c_in, c_out, hw, k, s, p):
    rng = np.random.default_rng(c_in * 1000 + c_out * 10 + k)
    sp = _spec(dtype, c_in, hw, c_out, k, s, p, rng)
    video = _video(dtype, c_in, hw, 5, 2, rng)
    _run([sp], video, n=2, stats=True)


@pytest.mark.parametrize("dtype", ["f32", "i8", "bin"])
@pytest.mark.parametrize("c_in,c_out,hw,k,s,p,n", [
    (32, 64, (11, 10), 3, 1, 1, 1),          # one accumulator tile, K cut into parts of one block's taps
    (160, 130, (8, 9), 3, 1, 1, 2),          # ragged blocks of K groups, two column tiles of uneven width
    (24, 33, (30, 31), 3, 2, 1, 3),          # stride 2: four planes; rows that are no multiple of 16 bytes
    (20, 16, (25, 23), 5, 3, 2, 1),          # stride 3: nine planes, some with fewer taps
    (16, 20, (140, 139), 3, 1, 1, 2),        # enough rows for two accumulator tiles per thread block
    (2, 72, (41, 38), 9, 4, 3, 2),           # few channels, stride 4: the windows are image rows in one (int8) or two (fp32) arrays
    (3, 16, (45, 52), 9, 8, 2, 1),           # ... stride 8: in two (int8), or column by column (fp32)
    (12, 24, (3, 1400), 3, 1, 1, 1)])        # a window wider than shared memory takes: the other kernels
def test_window_convolution_tile_edges(dtype, c_in, c_out, hw, k, s, p, n, monkeypatch):
    rng = np.random.default_rng(c_in * 1000 + c_out * 10 + k)
    sp = _spec(dtype, c_in, hw, c_out, k, s, p, rng)
    video = _video(dtype, c_in, hw, 5, n, rng)
    _run([sp], video, n=n, stats=True, keyframe_at=(4,))
    # the same frames as one chunk, every kernel taking all of them
    monkeypatch.setenv("RRM_CHUNK_BY_LAYER", "1")
    net = _rrm().net_from_specs([sp], n=n)
    net.set_options(chunk_dense_activity=2.0, stack_dense_activity=2.0)
    outs = net.new_output(frames=5)
    net.step_seq(torch.stack([_frame_to_dev([sp], f) for f in video]), outs, 5)
    for t in range(5):
        want = orc.dense_forward([sp], video[t])[0][1]
        got = outs[t].cpu().numpy()
        if dtype == "f32":
            assert float(np.abs(got - want).max()) <= F32_TOL * float(np.abs(want).max()), t
        else:
            np.testing.assert_array_equal(got.astype(np.int64), want, err_msg=f"frame {t}")
    _compare([sp], net, video[4], 4)
    net.close()


@pytest.mark.parametrize("dtype", ["f32", "i8"])
@pytest.mark.parametrize("hw,k,s,p,n", [
    ((601, 18), 5, 4, 2, 1),                 # planes as rows further down: more rows left than the table counts, the last plane one row short
    ((256, 17), 7, 2, 3, 2)])                # ... and exactly one more than it counts
def test_first_layer_tables_of_tall_images(dtype, hw, k, s, p, n):
    rng = np.random.default_rng(hw[0] + k)
    sp = _spec(dtype, 3, hw, 20, k, s, p, rng)
    _run([sp], _video(dtype, 3, hw, 4, n, rng), n=n, stats=True, keyframe_at=(3,))


@pytest.mark.parametrize("c_in,c_out,hw,k,s,p", [
    (3, 8, (480, 640), 7, 2, 3), (3, 8, (300, 512), 3, 1, 1), (2, 4, (1080, 1920), 11, 4, 0),      # first layers
    (16, 8, (240, 470), 3, 1, 1)])                                                                 # ... and one of more channels
def test_windows_of_wide_images_fit_their_tables(c_in, c_out, hw, k, s, p):
    """int8 layers large enough for two accumulator tiles per thread block whose window fits the kernel's per-pixel tables
    with one tile only (a span of 1025 to 1152 pixels): frame by frame, as a keyframe and in a dense chunk."""
    rng = np.random.default_rng(hw[1] + k)
    sp = _spec("i8", c_in, hw, c_out, k, s, p, rng)
    video = _video("i8", c_in, hw, 4, 1, rng)
    video[2:] = video[1]                                      # a patch at the image's far corner, one in its middle
    video[2, :, :, -9:, -9:] ^= 1
    video[3, :, :, hw[0] // 2:hw[0] // 2 + 9, hw[1] // 2:hw[1] // 2 + 9] ^= 3
    net = _rrm().net_from_specs([sp])
    out, outs = net.new_output(), net.new_output(frames=2)
    want = [orc.dense_forward([sp], f)[0][1] for f in video[1:]]
    for t, call in ((1, net.keyframe), (2, net.step), (3, net.step)):
        call(dev(video[t]), out)
        np.testing.assert_array_equal(out.cpu().numpy(), want[t - 1], err_msg=f"frame {t}")
    net.dense_seq(dev(video[2:4]), outs, 2)
    np.testing.assert_array_equal(outs.cpu().numpy(), np.stack(want[1:3]), err_msg="dense chunk")
    assert net.stats(0)["error_word"] == 0
    net.close()


@pytest.mark.parametrize("dtype,c_in,c_out,hw,n", [
    ("f32", 3, 40, (9, 15), 2), ("f32", 4, 8, (320, 300), 2),         # a thread per pixel; four pixel groups per thread
    ("f32", 64, 36, (13, 9), 2), ("f32", 8, 5, (6, 6), 3),            # 16 lanes per pixel: full, and few of them at work
    ("i8", 64, 33, (16, 16), 2), ("i8", 33, 70, (11, 13), 3),         # planes aligned to words, and not; ragged channel tiles
    ("i8", 96, 16, (17, 8), 1), ("i8", 3, 130, (33, 31), 2)])
def test_boundary_layouts(dtype, c_in, c_out, hw, n):
    """The kernels between the boundary layout and pixel rows: frames in, outputs out, frame by frame and in a dense
    chunk, at the edges of their tiles."""
    rng = np.random.default_rng(c_in * 100 + c_out)
    kw = dict(act="relu", shift=11) if dtype == "i8" else {}
    sp = _spec(dtype, c_in, hw, c_out, 1, 1, 0, rng, **kw)
    video = _video(dtype, c_in, hw, 5, n, rng)
    _run([sp], video, n=n, stats=True, keyframe_at=(4,))
    net = _rrm().net_from_specs([sp], n=n)
    outs = net.new_output(frames=3)
    net.dense_seq(dev(video[1:4]), outs, 3)
    for t in range(3):
        want = orc.dense_forward([sp], video[1 + t])[0][1]
        got = outs[t].cpu().numpy()
        if dtype == "f32":
            assert float(np.abs(got - want).max()) <= F32_TOL * float(np.abs(want).max()), t
        else:
            np.testing.assert_array_equal(got.astype(np.int64), want, err_msg=f"frame {t}")
    net.close()


@pytest.mark.parametrize("c_in,hw,n", [(1, (9, 7), 1), (2, (5, 5), 3), (3, (7, 9), 4), (3, (33, 41), 3), (4, (6, 11), 2), (3, (2, 1), 5)])
def test_dense_frames_of_few_channels_start_anywhere(c_in, hw, n):
    """Keyframes of int8 frames of up to 4 channels, at every alignment of the frame's first byte: pixels of two images in one
    thread, planes whose bytes straddle words, the first and last words."""
    rng = np.random.default_rng(c_in * hw[1])
    sp = _spec("i8", c_in, hw, 8, 1, 1, 0, rng, act="relu", shift=6)
    net = _rrm().net_from_specs([sp], n=n)
    for off in range(4):
        x = rng.integers(-127, 128, size=(n, c_in) + hw).astype(np.int8)
        raw = torch.zeros(x.size + 4, dtype=torch.int8, device="cuda")
        frame = raw[off:off + x.size].view(n, c_in, *hw)
        frame.copy_(torch.from_numpy(x))
        net.keyframe(frame)
        _compare([sp], net, x, off)
    net.close()


@pytest.mark.parametrize("dtype,n,T", [("i8", 512, 1), ("i8", 16, 32), ("f32", 512, 1), ("f32", 16, 32)])
def test_boundary_layouts_of_many_streams_of_many_channels(dtype, n, T):
    """Channel tiles x streams x frames of a launch at 65536, one more than a grid has along y: 4096 channels in (int8) and out."""
    rng = np.random.default_rng(n + T)
    dims = [(4096, 32), (32, 4096)] if dtype == "i8" else [(16, 4096)]
    specs = []
    for l, (a, b) in enumerate(dims):
        kw = dict(act="relu", shift=12) if dtype == "i8" else {}
        sp = _spec(dtype, a, (1, 1), b, 1, 1, 0, rng, **kw)
        sp.src = l
        specs.append(sp)
    shape = (T, n, dims[0][0], 1, 1)
    frames = rng.integers(0, 128, size=shape).astype(np.int8) if dtype == "i8" else rng.standard_normal(shape).astype(np.float32)
    net = _rrm().net_from_specs(specs, n=n)
    if T == 1:
        outs = net.new_output()
        net.keyframe(dev(frames[0]), outs)
        got = [outs.cpu().numpy()]
    else:
        outs = net.new_output(frames=T)
        net.dense_seq(dev(frames), outs, T)
        got = outs.cpu().numpy()
    for t in range(0, T, 31):
        want = orc.dense_forward(specs, frames[t])[0][-1]
        if dtype == "f32":
            assert float(np.abs(got[t] - want).max()) <= F32_TOL * float(np.abs(want).max()), t
        else:
            np.testing.assert_array_equal(got[t].astype(np.int64), want, err_msg=f"frame {t}")
    net.close()


@pytest.mark.parametrize("c_in,c_out,hw,k,s,p,n", [(4, 162, (19, 77), 11, 1, 3, 2), (3, 64, (64, 1110), 9, 3, 0, 1)])
def test_first_layers_whose_window_leaves_room_for_one_tile_width(c_in, c_out, hw, k, s, p, n):
    """A window beside which only the stages of 96 columns fit, and one beside which only those of 32 do: keyframes, steps and dense
    chunks."""
    rng = np.random.default_rng(c_out)
    sp = _spec("i8", c_in, hw, c_out, k, s, p, rng, act="relu", shift=9)
    video = _video("i8", c_in, hw, 4, n, rng)
    _run([sp], video, n=n, keyframe_at=(1,))
    net = _rrm().net_from_specs([sp], n=n)
    outs = net.new_output(frames=4)
    net.dense_seq(torch.from_numpy(video).cuda(), outs)
    for t in range(4):
        np.testing.assert_array_equal(outs[t].cpu().numpy().astype(np.int64), orc.dense_forward([sp], video[t])[0][1], err_msg=f"frame {t}")
    net.close()


@pytest.mark.parametrize("dtype", ["i8", "bin"])
@pytest.mark.parametrize("c_in,c_out,hw,k,s,p,n,dense,delta", [
    # (columns, accumulator tiles per CTA, shares): one share (18 and 90 K steps), ragged columns
    (64, 70, (14, 13), 3, 1, 1, 1, (32, 1, 1), (32, 1, 1)), (320, 200, (13, 13), 3, 1, 1, 1, (32, 1, 1), (128, 1, 10)),
    # clusters of 2, strides, deltas in clusters; a layer whose shares of wide tiles are ahead
    (352, 130, (9, 11), 3, 1, 1, 2, (32, 1, 2), (96, 1, 6)), (96, 96, (17, 18), 5, 2, 2, 3, (32, 1, 8), (96, 1, 12)),
    (512, 64, (7, 7), 3, 1, 1, 4, (64, 1, 8), (64, 1, 16)), (32, 33, (8, 8), 1, 1, 0, 1, (32, 1, 1), (32, 1, 1)),
    # 74 and 75 wide tiles; 74 of 128 columns are 296 narrow ones, of which a CTA takes two
    (32, 64, (96, 97), 3, 1, 1, 1, (32, 1, 1), (64, 1, 2)), (32, 64, (97, 97), 3, 1, 1, 1, (64, 1, 1), (64, 1, 1)),
    (32, 256, (12, 12), 3, 1, 1, 28, (32, 2, 1), (128, 1, 2)), (32, 250, (12, 12), 3, 1, 1, 28, (32, 2, 1), (32, 2, 1)),
    # first layers (binary ones are not), of wide windows too
    (3, 96, (60, 61), 11, 4, 0, 1, {"i8": (32, 1, 4), "bin": (32, 1, 8)}, {"i8": (96, 1, 4), "bin": (96, 1, 16)}),
    (3, 96, (24, 500), 7, 2, 3, 1, {"i8": (32, 1, 2), "bin": (96, 1, 4)}, {"i8": (96, 1, 2), "bin": (96, 1, 4)})])
def test_dense_passes_of_few_tiles_take_narrow_ones(dtype, c_in, c_out, hw, k, s, p, n, dense, delta):
    """Keyframes and dense passes whose tiles would leave the machine idle run as tiles of 32 columns; with f in the kernel
    (int8, signs), as raw projections, and with delta steps in between."""
    rng = np.random.default_rng(c_in + c_out)
    for kw in ((dict(act="sign", theta=1), dict(shift=-1, act="none")) if dtype == "bin" else (dict(act="relu", shift=8), dict(shift=-1, act="none"))):
        sp = _spec(dtype, c_in, hw, c_out, k, s, p, rng, **kw)
        for form, want in (("dense", dense), ("delta", delta)):
            got = _rrm().plan_conv(_rrm().desc_from_spec(sp, n), form)
            assert (got["columns"], got["tiles_per_cta"], got["shares"]) == (want[dtype] if isinstance(want, dict) else want), (form, got)
        _run([sp], _video(dtype, c_in, hw, 4, n, rng), n=n, stats=n < 28, keyframe_at=(1, 3))


@pytest.mark.parametrize("c_in,c_out,hw,k,s,p,n,plan", [
    (420, 33, (20, 19), 3, 3, 0, 3, (32, 1, 8)),             # clusters; a last block of two of four groups
    (70, 128, (34, 31), 3, 2, 1, 8, (32, 1, 1)), (512, 70, (14, 13), 1, 1, 0, 2, (32, 1, 1)),      # narrow tiles; one plane
    (260, 40, (61, 60), 3, 3, 1, 9, (64, 1, 4)), (32, 64, (41, 40), 3, 2, 1, 92, (64, 2, 1))])     # two accumulator tiles
def test_dense_windows_of_many_short_blocks(c_in, c_out, hw, k, s, p, n, plan):
    """Dense int8 passes whose windows come by asynchronous copies, as outputs and as raw projections, delta steps in between."""
    rng = np.random.default_rng(c_in + c_out)
    for kw in (dict(act="relu", shift=8), dict(shift=-1, act="none")):
        sp = _spec("i8", c_in, hw, c_out, k, s, p, rng, **kw)
        got = _rrm().plan_conv(_rrm().desc_from_spec(sp, n), "dense")
        assert got["async_windows"] and (got["columns"], got["tiles_per_cta"], got["shares"]) == plan, got
        _run([sp], _video("i8", c_in, hw, 4, n, rng), n=n, keyframe_at=(1, 3))


def _dense_outputs(path):
    """Keyframes, dense passes and dense chunks of three stacks and of layers whose launches lie alone on their SMs or are not
    launched early; every call twice in a row, so that a pass starts while the last one ends."""
    rrm, got = _rrm(), {}
    rng = np.random.default_rng(8)
    nets = [("f32", wl.alexnet_convs("f32", hw=67), 2, (3, 67, 67)), ("i8", wl.alexnet_convs("i8", hw=67), 3, (3, 67, 67)),
            ("bin", wl.xnor_alexnet_convs(hw=67), 2, (3, 67, 67)), ("res", wl.resnet18_convs(hw=64), 2, (3, 64, 64))]
    for i, (dtype, c_in, c_out, hw, k, s, p, n) in enumerate((
            ("bin", 411, 22, (27, 37), 3, 2, 1, 56), ("bin", 457, 69, (84, 68), 3, 3, 0, 11), ("i8", 64, 64, (56, 56), 3, 1, 1, 4),
            ("i8", 212, 163, (15, 15), 9, 2, 0, 12), ("i8", 73, 296, (17, 9), 7, 1, 0, 1), ("f32", 130, 150, (22, 15), 7, 1, 0, 7), ("f32", 162, 105, (18, 20), 7, 3, 0, 6))):
        nets.append((f"{dtype}{i}", [_spec(dtype, c_in, hw, c_out, k, s, p, rng, **(dict(act="sign", theta=1) if dtype == "bin" else dict(act="relu", shift=9)))],
                     n, (c_in,) + hw))
    for name, specs, n, shape in nets:
        net = rrm.net_from_specs(specs, n=n)
        x = _frame_to_dev(specs, _video(specs[0].dtype, shape[0], shape[1:], 4, n, rng)[0])
        y = x.flip(0).contiguous()
        out, outs = net.new_output(), net.new_output(frames=3)
        for what in ("keyframe", "dense"):
            getattr(net, what)(x, out)
            getattr(net, what)(y, out)
            got[f"{name} {what}"] = out.cpu().numpy()
        for _ in range(2):
            net.dense_seq(torch.stack((x, y, x)), outs)
        got[f"{name} chunk"] = outs.cpu().numpy()
        net.close()
    np.savez(path, **got)


def test_dense_launches_that_overlap_give_the_same_bits(tmp_path):
    """With the launches of dense passes overlapping their predecessors, and (in a process of its own: the switch is read once)
    without."""
    _dense_outputs(tmp_path / "overlapping.npz")
    code = f"import sys; sys.path[:0] = [{os.path.dirname(__file__)!r}, {os.path.dirname(os.path.dirname(__file__))!r}]; import test_gpu_conv as t; t._dense_outputs({str(tmp_path / 'apart.npz')!r})"
    subprocess.run([sys.executable, "-c", code], check=True, timeout=600, env=dict(os.environ, RRM_PDL="0"))
    a, b = np.load(tmp_path / "overlapping.npz"), np.load(tmp_path / "apart.npz")
    assert sorted(a.files) == sorted(b.files) and len(a.files) == 33
    for name in a.files:
        np.testing.assert_array_equal(a[name], b[name], err_msg=name)


@pytest.mark.parametrize("dtype", ["f32", "i8", "bin"])
@pytest.mark.parametrize("c_in,c_out,hw,k,s,p,pool", [
    (24, 20, (5, 700), 3, 1, 1, (3, 2, 0)),  # wider than 510 pixels
    (16, 33, (4, 2300), 3, 2, 1, None),      # ... than 2040 at stride 2
    (40, 70, (7, 7), 7, 1, 0, None),         # a filter that covers the map: more zeros than pixels in a window
    (3, 12, (6, 300), 5, 1, 2, (2, 2, 0))])  # a first layer, 5x5, wider than 250
def test_layers_beyond_the_window_kernel(dtype, c_in, c_out, hw, k, s, p, pool, monkeypatch):
    """What the window convolution does not take runs in the kernel that gathers compacted rows (int8, binary) or on the
    CUDA cores (fp32): frame by frame, as keyframes, and as chunks of both forms."""
    rng = np.random.default_rng(hw[1] + k)
    kw = dict(pool=pool) if dtype == "f32" else dict(act="sign", theta=2, pool=pool) if dtype == "bin" else dict(act="relu", shift=9, pool=pool)
    sp = _spec(dtype, c_in, hw, c_out, k, s, p, rng, **kw)
    video = _video(dtype, c_in, hw, 6, 2, rng)
    _run([sp], video, n=2, stats=True, keyframe_at=(4,))
    for form in ("RRM_CHUNK_BY_LAYER", "RRM_CHUNK_PIPELINED"):
        monkeypatch.delenv("RRM_CHUNK_BY_LAYER", raising=False)
        monkeypatch.setenv(form, "1")
        net = _rrm().net_from_specs([sp], n=2)
        net.keyframe(_frame_to_dev([sp], video[0]))
        net.step_seq(torch.stack([_frame_to_dev([sp], f) for f in video[1:]]), net.new_output(frames=5), 5)
        _compare([sp], net, video[5], 5)
        net.close()
    monkeypatch.delenv("RRM_CHUNK_PIPELINED")
    net = _rrm().net_from_specs([sp], n=2)
    dense, one = net.new_output(frames=6), net.new_output()
    net.dense_seq(torch.stack([_frame_to_dev([sp], f) for f in video]), dense, 6)
    for t in range(6):
        net.keyframe(_frame_to_dev([sp], video[t]), one)
        _compare([sp], net, video[t], t)
        if dtype == "f32":
            assert float((dense[t] - one).abs().max()) <= F32_TOL * float(one.abs().max())
        else:
            assert torch.equal(dense[t], one), t
    net.close()


# fp32 sums against fp64, 2-norm: measured up to 4.0e-7 on the layers below (chains of fused multiply-adds on the CUDA cores:
# 4.2e-7), twice that here.  Without the third bf16 piece of the operands the tensor-core kernels would be at 3.4e-6, without the
# promoted sums at 1.7e-6.
F32_REL = 8e-7


@pytest.mark.parametrize("exp_x,exp_w", [(0, 0), (-110, 100), (100, -110)])
@pytest.mark.parametrize("c_in,c_out,hw,k,s,p,n", [
    (3, 40, (47, 51), 11, 4, 0, 1), (4, 16, (200, 180), 3, 1, 1, 1),          # first layers
    (64, 48, (20, 21), 3, 1, 1, 1), (256, 130, (13, 13), 3, 1, 1, 1), (512, 64, (30, 30), 3, 2, 1, 2),
    (1500, 32, (1, 1), 1, 1, 0, 40)])
def test_fp32_layers_keep_fp32_accuracy(c_in, c_out, hw, k, s, p, n, exp_x, exp_w):
    """Values over twenty powers of two, near one and near the ends of the exponent range, dense and as deltas."""
    rng = np.random.default_rng(c_in + k)
    sp = _spec("f32", c_in, hw, c_out, k, s, p, rng)
    sp.weight = np.ldexp(sp.weight, exp_w).astype(np.float32)
    sp.bias = np.ldexp(sp.bias, exp_x + exp_w).astype(np.float32)
    shape = (3, n, c_in) + hw
    video = np.ldexp(rng.standard_normal(shape) * np.exp2(rng.uniform(-10, 10, size=shape)), exp_x).astype(np.float32)
    video[1:] = np.where(rng.random((2, n, 1) + hw) < 0.3, video[1:], video[0])
    net = _rrm().net_from_specs([sp], n=n)
    for t, call in enumerate((net.keyframe, net.step, net.step)):
        call(dev(video[t]))
        want = orc.dense_forward([sp], video[t])[1][0]
        err = np.linalg.norm(net.projection(0).cpu().numpy().astype(np.float64) - want) / np.linalg.norm(want)
        assert err <= F32_REL, (t, err)
    net.close()


@pytest.mark.parametrize("c_in,c_out,hw,k,s,p", [
    (3, 16, (60, 61), 7, 2, 3), (3, 20, (40, 44), 5, 4, 2),                   # first layers: windows of more columns than the filter has
    (20, 24, (12, 11), 3, 1, 1), (64, 70, (90, 91), 3, 1, 1)])                # a cluster of shares; shares of their own
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 3.4e38, -3.399e38])
def test_fp32_values_without_bf16_pieces(c_in, c_out, hw, k, s, p, value):
    """Infinities, NaNs and floats above bf16's largest reach the outputs that see them, as in fp32 arithmetic, and no others."""
    rng = np.random.default_rng(c_in + k)
    sp = _spec("f32", c_in, hw, c_out, k, s, p, rng)
    video = rng.standard_normal((2, 1, c_in) + hw).astype(np.float32)
    video[1] = video[0]
    video[1, 0, 1, hw[0] // 2, hw[1] // 2] = value
    video[1, 0, 0, 0, hw[1] - 1] = value
    net = _rrm().net_from_specs([sp])
    with np.errstate(all="ignore"):
        plain = orc.dense_forward([sp], video[0])[1][0]
        want = orc.dense_forward([sp], video[1])[1][0]
        want = np.where(np.abs(want) > np.finfo(np.float32).max, np.copysign(np.inf, want), want)

    def check(got, what):
        np.testing.assert_array_equal(np.isnan(got), np.isnan(want), err_msg=what)
        np.testing.assert_array_equal(np.isinf(got) * np.sign(got), np.isinf(want) * np.sign(want), err_msg=what)
        fin = np.isfinite(want)
        assert np.all(np.abs(got[fin] - want[fin]) <= F32_TOL * np.maximum(np.abs(plain).max(), np.abs(want[fin]))), what

    out, outs = net.new_output(), net.new_output(frames=2)
    net.keyframe(dev(video[1]), out)
    check(out.cpu().numpy().astype(np.float64), "keyframe")
    net.dense_seq(dev(video), outs, 2)
    check(outs[1].cpu().numpy().astype(np.float64), "dense chunk")
    net.keyframe(dev(video[0]), out)
    net.step(dev(video[1]), out)
    check(out.cpu().numpy().astype(np.float64), "step")
    # ... and a filter value of that kind (the middle one: it meets no padding)
    sp.weight[1, 1, k // 2, k // 2] = value
    net2 = _rrm().net_from_specs([sp])
    with np.errstate(all="ignore"):
        want = orc.dense_forward([sp], video[0])[1][0]
        want = np.where(np.abs(want) > np.finfo(np.float32).max, np.copysign(np.inf, want), want)
    net2.keyframe(dev(video[0]), out)
    check(out.cpu().numpy().astype(np.float64), "filter")
    net.close()
    net2.close()


@pytest.mark.parametrize("dtype", ["i8", "bin"])
@pytest.mark.parametrize("c_in,c_out,hw,k,s,p", [(16, 70, (13, 13), 3, 1, 1), (8, 12, (17, 15), 5, 2, 2), (64, 16, (10, 10), 3, 1, 1),
                                                 (3, 6, (35, 35), 11, 4, 0)])
def test_single_layer_cuda_core_variant(dtype, c_in, c_out, hw, k, s, p):
    """The CUDA-core (dp4a / popcount) variant on layers that would otherwise take the tensor-core one."""
    rng = np.random.default_rng(c_in * 1000 + c_out * 10 + k + 1)
    sp = _spec(dtype, c_in, hw, c_out, k, s, p, rng)
    video = _video(dtype, c_in, hw, 5, 2, rng)
    _run([sp], video, n=2, stats=True, variant="gather")


@pytest.mark.parametrize("dtype,act,pool,shift", [
    ("f32", "relu", (3, 2, 0), -1), ("f32", "relu", (3, 2, 1), -1), ("f32", "none", (2, 2, 0), -1),
    ("f32", "leaky", None, -1), ("f32", "leaky", (2, 2, 0), -1),
    ("i8", "relu", (3, 2, 0), 9), ("i8", "none", None, 10), ("i8", "sign", (3, 2, 0), -1), ("i8", "none", (3, 2, 1), -1),
    ("bin", "sign", None, -1), ("bin", "sign", (3, 2, 0), -1), ("bin", "none", (3, 2, 0), -1)])
def test_single_layer_nonlinearities(dtype, act, pool, shift):
    rng = np.random.default_rng(77)
    sp = _spec(dtype, 12, (15, 14), 40, 3, 1, 1, rng, act=act, pool=pool, shift=shift, theta=3)
    video = _video(dtype, 12, (15, 14), 5, 1, rng)
    _run([sp], video, n=1, stats=True)


def test_keyframe_resets_state_and_dense_path_is_stateless():
    rrm = _rrm()
    specs = wl.single_conv_f32(c_in=8, c_out=8, hw=20)
    video = wl.block_redraw_sequence(frames=6, c=8, hw=20, seed=3)
    _run(specs, video, keyframe_at=(0, 3))
    net = rrm.net_from_specs(specs)
    out, outd = net.new_output(), net.new_output()
    net.step(dev(video[0]), out)
    net.dense(dev(video[4]), outd)
    ref = orc.dense_forward(specs, video[4])[0][1]
    assert np.abs(outd.cpu().numpy() - ref).max() <= F32_TOL * np.abs(ref).max()
    net.step(dev(video[1]), out)
    ref = orc.dense_forward(specs, video[1])[0][1]
    assert np.abs(out.cpu().numpy() - ref).max() <= F32_TOL * np.abs(ref).max()
    net.close()


# ------------------------------------------------------------------ small stacks, every frame, with stats
@pytest.mark.parametrize("name", ["alex_f32", "alex_i8", "resnet_i8", "xnor"])
def test_small_stacks_every_frame(name):
    if name == "alex_f32":
        specs, dt, hw = wl.alexnet_convs("f32", hw=99, scale=8), "f32", 99
    elif name == "alex_i8":
        specs, dt, hw = wl.alexnet_convs("i8", hw=99, scale=8), "i8", 99
    elif name == "resnet_i8":
        specs, dt, hw = wl.resnet18_convs(hw=96, scale=8), "i8", 96
    else:
        specs, dt, hw = wl.xnor_alexnet_convs(hw=99, scale=8), "i8", 99
    n = 2 if name == "resnet_i8" else 1
    video = wl.moving_rect_video(frames=6, hw=hw, dtype=dt, seed=9, n=n, side=(12, 24),
                                 bg_redraw=0.02 if name == "resnet_i8" else 0.0)
    _run(specs, video, n=n, stats=True, keyframe_at=(4,))


# ------------------------------------------------------------------ whole networks: FC layers inside a stack, VGG-16 shape
@pytest.mark.parametrize("name", ["alexnet_full_i8", "alexnet_full_f32", "vgg16_i8", "vgg16_f32"])
def test_second_workloads_every_frame(name):
    dt = "i8" if name.endswith("i8") else "f32"
    if name.startswith("alexnet_full"):
        specs, hw = wl.alexnet_full(dt, hw=99, scale=8, classes=80), 99
    else:
        specs, hw = wl.vgg16_convs(dt, hw=64, scale=8), 64
    video = wl.moving_rect_video(frames=5, hw=hw, dtype=dt, seed=12, side=(10, 20))
    _run(specs, video, stats=True, keyframe_at=(3,))


def test_large_stack_goes_dense_while_nearly_every_pixel_changes():
    """Background noise makes every projection pixel change: after the first measured delta frame the frames
    are evaluated densely (same results), with a delta frame every 16th frame to measure again."""
    rrm = _rrm()
    specs = wl.alexnet_convs("i8")
    video = wl.moving_rect_video(frames=20, hw=227, dtype="i8", seed=33, n=2, bg_redraw=0.10)
    net = rrm.net_from_specs(specs, n=2)
    out = net.new_output()
    variants, counted = [], []
    for t in range(20):
        net.step(dev(video[t]), out)
        st = net.stats(1)                     # synchronises, so the next call sees this frame's counters
        variants.append(st["variant"])
        counted.append(st["nnz_elems"] != -1)
        if t in (0, 1, 2, 16, 19):
            _compare(specs, net, video[t], t)
    assert variants[0] == 2 and counted[0]                # the first frame (every pixel new) is a measured delta frame
    assert all(v == 3 for v in variants[1:16]) and not any(counted[1:16])   # the whole stack dense while the measured activity is high
    # one delta frame measures again (the per-layer choice is off by default: its layers run the sparse product)
    assert variants[16] == 2 and counted[16]
    assert variants[17] == 3 and not counted[17]
    net.close()


@pytest.mark.parametrize("name", ["alex_i8", "resnet_i8", "alex_f32", "xnor"])
def test_layers_choose_between_sparse_and_dense_evaluation_from_their_measured_activity(name):
    """Per-layer choice (variant AUTO): with the thresholds lowered, the layers whose share of projection pixels to
    update is high run a dense evaluation inside the delta step while the others run the sparse product.  Outputs,
    stored projections and counters stay those of Algorithm 1 at every frame, whatever the mix."""
    rrm = _rrm()
    if name == "alex_i8":
        specs, dt, hw, n = wl.alexnet_convs("i8", hw=99, scale=8), "i8", 99, 1
    elif name == "resnet_i8":
        specs, dt, hw, n = wl.resnet18_convs(hw=96, scale=8), "i8", 96, 2
    elif name == "alex_f32":
        specs, dt, hw, n = wl.alexnet_convs("f32", hw=99, scale=8), "f32", 99, 1
    else:
        specs, dt, hw, n = wl.xnor_alexnet_convs(hw=99, scale=8), "i8", 99, 1
    video = wl.moving_rect_video(frames=9, hw=hw, dtype=dt, seed=23, n=n, side=(12, 24))
    net = rrm.net_from_specs(specs, n=n)
    rec = orc.Recurrence(specs, n=n)
    rec.step(np.full_like(video[0], 0))
    out = net.new_output()
    mixes = set()
    for t in range(video.shape[0]):
        net.step(dev(video[t]), out)
        rec.step(video[t])
        vs, acts = [], []
        for l in range(len(specs)):
            st = net.stats(l)                 # synchronises: the next step's choice sees this frame's counters
            vs.append(st["variant"])
            acts.append(st["active_out_pixels"] / st["out_pixels"])
            assert st["error_word"] == 0
            if dt != "f32" or l == 0:
                assert st["nnz_elems"] == rec.nnz[l] and st["active_macs"] == rec.macs[l], (t, l, st, rec.nnz[l], rec.macs[l])
        mixes.add(tuple(v == 3 for v in vs))
        _compare(specs, net, video[t], t)
        if t == 2:
            # thresholds between this video's measured per-layer activities, so that the layers really split
            a = sorted(set(acts))
            assert len(a) >= 2, acts
            thr = 0.5 * (a[len(a) // 2 - 1] + a[len(a) // 2])
            net.set_options(layer_dense_activity=thr, layer_delta_activity=0.95 * thr)
    assert any(any(m) and not all(m) for m in mixes), mixes       # some frame ran a real mix of the two evaluations
    # ... and a chunk of frames with the mix chosen at its start
    more = wl.moving_rect_video(frames=13, hw=hw, dtype=dt, seed=23, n=n, side=(12, 24))
    outs = net.new_output(frames=4)
    net.step_seq(dev(np.ascontiguousarray(more[9:13])), outs, 4)
    _compare(specs, net, more[12], 12)
    net.close()


# ------------------------------------------------------------------ full-size configs, sampled frames
def test_cfg3_alexnet_fp32_full_size():
    specs = wl.alexnet_convs("f32")
    video = wl.moving_rect_video(frames=64, hw=227, dtype="f32", seed=31)
    _run(specs, video, check_frames={0, 1, 2, 17, 63})


def test_cfg3_alexnet_int8_full_size():
    specs = wl.alexnet_convs("i8")
    video = wl.moving_rect_video(frames=64, hw=227, dtype="i8", seed=32)
    _run(specs, video, check_frames={0, 1, 30, 63}, stats_frames={30})


def test_cfg3_alexnet_int8_early_layers_sparse_late_layers_dense():
    """On the moving-rectangle video the first layers update a fifth to a half of their projection pixels, the last
    ones nearly all: with the thresholds at 0.75 / 0.60 the library settles on the sparse product for conv1-2 and a
    dense evaluation for conv5, inside the same delta step."""
    rrm = _rrm()
    specs = wl.alexnet_convs("i8")
    video = wl.moving_rect_video(frames=20, hw=227, dtype="i8", seed=32)
    net = rrm.net_from_specs(specs)
    net.set_options(layer_dense_activity=0.75, layer_delta_activity=0.60)
    out = net.new_output()
    # (frame 0 changes every pixel, so this stack of > 1 GMAC is evaluated densely as a whole for the next 15 frames;
    # frame 16 measures again, and from frame 17 on every layer follows its own activity)
    for t in range(20):
        net.step(dev(video[t]), out)
        vs = [net.stats(l)["variant"] for l in range(len(specs))]
    assert vs[0] == 2 and vs[1] == 2 and vs[4] == 3, vs
    act = [net.stats(l)["active_out_pixels"] / net.stats(l)["out_pixels"] for l in range(len(specs))]
    assert act[0] < 0.6 and act[4] > 0.75, act
    _compare(specs, net, video[19], 19)
    net.close()


def test_cfg4_resnet18_int8_batch4():
    specs = wl.resnet18_convs()
    video = wl.moving_rect_video(frames=64, hw=224, dtype="i8", seed=41, n=4, bg_redraw=0.02)
    _run(specs, video, n=4, check_frames={0, 1, 63})


def test_cfg4_resnet18_int8_batch4_every_frame_through_the_delta_kernels():
    """The same stack with the delta / dense switch off (variant "tensor"): every frame goes through the sparse
    product at partial density, every layer's projection is compared at five frames, the counters at two."""
    specs = wl.resnet18_convs()
    video = wl.moving_rect_video(frames=64, hw=224, dtype="i8", seed=41, n=4, bg_redraw=0.02)
    _run(specs, video, n=4, check_frames={0, 1, 16, 32, 63}, stats_frames={16, 63}, variant="tensor")


def test_cfg5_xnor_alexnet_128_frames():
    specs = wl.xnor_alexnet_convs()
    video = wl.moving_rect_video(frames=128, hw=227, dtype="i8", seed=51)
    _run(specs, video, check_frames={0, 1, 64, 127}, stats_frames={64})


# ------------------------------------------------------------------ chunks of frames through a stack (frames overlap layer by layer)
@pytest.mark.parametrize("by_layer", [False, True])
@pytest.mark.parametrize("name", ["alex_f32", "alex_i8", "resnet_i8", "xnor", "alexnet_full_i8"])
def test_stack_chunks_of_frames_equal_frame_by_frame(name, by_layer, monkeypatch):
    """rrm_net_step_seq on a stack runs the frames of a chunk as one graph in which consecutive frames overlap, or
    (by_layer: forced here, chosen by the library for long chunks of few streams) every layer over all frames of the
    chunk in one launch; every frame's output, the state after each chunk and the last frame's counters are those of
    Algorithm 1."""
    if by_layer:
        monkeypatch.setenv("RRM_CHUNK_BY_LAYER", "1")
    rrm = _rrm()
    if name == "alex_f32":
        specs, dt, hw = wl.alexnet_convs("f32", hw=99, scale=8), "f32", 99
    elif name == "alex_i8":
        specs, dt, hw = wl.alexnet_convs("i8", hw=99, scale=8), "i8", 99
    elif name == "resnet_i8":
        specs, dt, hw = wl.resnet18_convs(hw=96, scale=8), "i8", 96
    elif name == "xnor":
        specs, dt, hw = wl.xnor_alexnet_convs(hw=99, scale=8), "i8", 99
    else:
        specs, dt, hw = wl.alexnet_full("i8", hw=99, scale=8, classes=80), "i8", 99
    n = 2 if name == "resnet_i8" else 1
    video = wl.moving_rect_video(frames=17, hw=hw, dtype=dt, seed=19, n=n, side=(12, 24),
                                 bg_redraw=0.02 if name == "resnet_i8" else 0.0)
    net = rrm.net_from_specs(specs, n=n)
    rec = orc.Recurrence(specs, n=n)
    rec.step(np.full_like(video[0], 0))
    frames = dev(np.ascontiguousarray(video))
    t0 = 0
    for T in (5, 5, 2, 4):                    # the same length twice (graph reuse), then other lengths
        outs = net.new_output(frames=T)
        net.step_seq(frames[t0:t0 + T], outs, T)
        for i in range(T):
            rec.step(video[t0 + i])
            want = orc.dense_forward(specs, video[t0 + i])[0][len(specs)]
            got = outs[i].cpu().numpy()
            if dt == "f32":
                assert float(np.abs(got - want).max()) <= F32_TOL * max(1e-30, float(np.abs(want).max())), (t0 + i)
            elif _out_kind(specs[-1]) == "bin":
                np.testing.assert_array_equal(unpack_bits_nhwc(got.view(np.uint32), specs[-1].c_out), want, err_msg=f"frame {t0 + i}")
            else:
                np.testing.assert_array_equal(got.astype(np.int64), want, err_msg=f"frame {t0 + i}")
        t0 += T
        _compare(specs, net, video[t0 - 1], t0 - 1)          # every layer's stored projection and tensor after the chunk
        for l in range(len(specs)):
            st = net.stats(l)
            assert st["error_word"] == 0
            if dt != "f32" or l == 0:
                assert st["nnz_elems"] == rec.nnz[l] and st["active_macs"] == rec.macs[l], (t0, l, st)
    # frame-by-frame stepping carries on from the chunk's state
    out = net.new_output()
    net.step(dev(video[16]), out)
    _compare(specs, net, video[16], 16)
    # dense chunks leave the state alone
    outs = net.new_output(frames=3)
    net.dense_seq(frames[2:5], outs, 3)
    for i in range(3):
        want = orc.dense_forward(specs, video[2 + i])[0][len(specs)]
        got = outs[i].cpu().numpy()
        if dt == "f32":
            assert float(np.abs(got - want).max()) <= F32_TOL * max(1e-30, float(np.abs(want).max()))
        elif _out_kind(specs[-1]) == "bin":
            np.testing.assert_array_equal(unpack_bits_nhwc(got.view(np.uint32), specs[-1].c_out), want)
        else:
            np.testing.assert_array_equal(got.astype(np.int64), want)
    _compare(specs, net, video[16], 16)
    net.close()


@pytest.mark.parametrize("name", ["cfg1", "cfg3_f32", "cfg3_i8", "cfg5", "cfg4"])
def test_full_size_stacks_in_chunks_of_32_frames(name):
    """The full-size configurations in the launch configuration the bench times for chunks: 32 frames per
    rrm_net_step_seq call.  First chunk and second chunk on the delta path (thresholds out of reach), the third as the
    library chooses; sampled frames' outputs against the dense definition, every layer's state after each chunk, and
    the last frame's counters of the second chunk against Algorithm 1 brought to the frame before by a dense pass."""
    rrm = _rrm()
    n = 1
    if name == "cfg1":
        specs, dt, hw = wl.single_conv_f32(), "f32", 56
    elif name == "cfg3_f32":
        specs, dt, hw = wl.alexnet_convs("f32"), "f32", 227
    elif name == "cfg3_i8":
        specs, dt, hw = wl.alexnet_convs("i8"), "i8", 227
    elif name == "cfg5":
        specs, dt, hw = wl.xnor_alexnet_convs(), "i8", 227
    else:
        specs, dt, hw, n = wl.resnet18_convs(), "i8", 224, 4
    if name == "cfg1":
        video = wl.block_redraw_sequence(frames=96, seed=61)
    else:
        video = wl.moving_rect_video(frames=96, hw=hw, dtype=dt, seed=61, n=n, bg_redraw=0.02 if name == "cfg4" else 0.0)
    net = rrm.net_from_specs(specs, n=n)
    defaults = net.options()
    net.set_options(chunk_dense_activity=2.0, stack_dense_activity=2.0)
    frames = dev(np.ascontiguousarray(video))
    outs = net.new_output(frames=32)
    for k in range(3):
        if k == 2:
            net.set_options(chunk_dense_activity=defaults["chunk_dense_activity"], stack_dense_activity=defaults["stack_dense_activity"])
        net.step_seq(frames[32 * k:32 * k + 32], outs, 32)
        sts = [net.stats(l) for l in range(len(specs))]
        assert all(st["error_word"] == 0 for st in sts)
        for i in ((0, 13, 31) if k < 2 else (0, 31)):
            want = orc.dense_forward(specs, video[32 * k + i])[0][len(specs)]
            got = outs[i].cpu().numpy()
            if dt == "f32":
                assert float(np.abs(got - want).max()) <= F32_TOL * max(1e-30, float(np.abs(want).max())), (k, i)
            elif _out_kind(specs[-1]) == "bin":
                np.testing.assert_array_equal(unpack_bits_nhwc(got.view(np.uint32), specs[-1].c_out), want, err_msg=f"chunk {k} frame {i}")
            else:
                np.testing.assert_array_equal(got.astype(np.int64), want, err_msg=f"chunk {k} frame {i}")
        _compare(specs, net, video[32 * k + 31], 32 * k + 31)
        if k == 1:
            one = orc.Recurrence(specs, n=n)
            one.reset_to(video[62])
            one.step(video[63])
            for l, st in enumerate(sts):
                assert st["variant"] != 3 and st["nnz_elems"] != -1, (l, st)
                if dt != "f32" or l == 0:
                    assert st["nnz_elems"] == one.nnz[l] and st["active_macs"] == one.macs[l], (l, st, one.nnz[l], one.macs[l])
    net.close()


def test_large_stack_chunks_go_dense_while_nearly_every_pixel_changes():
    """The density switch of a large stack, chunk by chunk: the chunk after a measured high-activity delta chunk is
    evaluated densely (a sequence of precise inferences that replace the state); outputs and state stay exact."""
    rrm = _rrm()
    specs = wl.alexnet_convs("i8")
    video = wl.moving_rect_video(frames=13, hw=227, dtype="i8", seed=34, n=2, bg_redraw=0.10)
    net = rrm.net_from_specs(specs, n=2)
    frames = dev(np.ascontiguousarray(video))
    variants = []
    for k in range(3):
        outs = net.new_output(frames=4)
        net.step_seq(frames[4 * k:4 * k + 4], outs, 4)
        st = net.stats(1)                     # synchronises, so the next call sees this chunk's counters
        variants.append(st["variant"])
        assert (st["nnz_elems"] == -1) == (st["variant"] == 3)
        for i in (0, 3):
            want = orc.dense_forward(specs, video[4 * k + i])[0][len(specs)]
            np.testing.assert_array_equal(outs[i].cpu().numpy().astype(np.int64), want, err_msg=f"frame {4 * k + i}")
        _compare(specs, net, video[4 * k + 3], 4 * k + 3)
    assert variants[0] == 2 and variants[1] == 3 and variants[2] == 3, variants
    out = net.new_output()
    net.step(dev(video[12]), out)             # frame by frame from the state the dense chunks left
    _compare(specs, net, video[12], 12)
    net.close()


def test_long_chunks_of_a_tensor_core_stack_go_dense_from_the_measured_activity():
    """rrm_options.chunk_dense_activity: after a delta chunk that measured a high share of pixels to update, the next
    long chunks of an int8 stack are evaluated densely, batched over their frames; outputs and state stay exact, and
    with the threshold out of reach the library stays on the delta path."""
    rrm = _rrm()
    specs = wl.alexnet_convs("i8", hw=99, scale=8)
    video = wl.moving_rect_video(frames=65, hw=99, dtype="i8", seed=43, n=1, side=(12, 24), bg_redraw=0.10)
    net = rrm.net_from_specs(specs, n=1)
    assert abs(net.options()["chunk_dense_activity"] - 0.40) < 1e-6
    frames = dev(np.ascontiguousarray(video))
    variants = []
    for k in range(4):
        if k == 3:
            net.set_options(chunk_dense_activity=2.0)
        outs = net.new_output(frames=16)
        net.step_seq(frames[16 * k:16 * k + 16], outs, 16)
        st = net.stats(1)                     # synchronises, so the next call sees this chunk's counters
        variants.append(st["variant"])
        for i in (0, 7, 15):
            want = orc.dense_forward(specs, video[16 * k + i])[0][len(specs)]
            np.testing.assert_array_equal(outs[i].cpu().numpy().astype(np.int64), want, err_msg=f"frame {16 * k + i}")
        _compare(specs, net, video[16 * k + 15], 16 * k + 15)
    assert variants[0] != 3 and variants[1] == 3 and variants[2] == 3 and variants[3] != 3, variants
    out = net.new_output()
    net.step(dev(video[64]), out)
    _compare(specs, net, video[64], 64)
    net.close()


@pytest.mark.parametrize("dtype,T", [("i8", 7), ("i8", 8), ("f32", 8), ("bin", 9)])
def test_chunks_of_eight_frames_go_dense_by_their_accumulator_tiles(dtype, T):
    """Chunks of 8 or more frames go dense when most accumulator tiles hold a pixel to update, even with few pixels
    active; shorter ones stay on the delta path.  Every call has buffers of its own (the graph is pointed at them)."""
    rng = np.random.default_rng(T)
    sp = _spec(dtype, 40, (24, 23), 36, 3, 1, 1, rng)
    video = _video(dtype, 40, (24, 23), 1 + 3 * T, 2, rng)
    video[4:] = video[4]
    for t in range(5, video.shape[0]):                        # one small patch per frame and stream: few pixels, spread over the tiles
        y, x = int(rng.integers(0, 20)), int(rng.integers(0, 19))
        video[t] = video[t - 1]
        video[t, :, :, y:y + 4, x:x + 4] = video[2, :, :, x:x + 4, y:y + 4] if dtype != "bin" else -video[t - 1, :, :, y:y + 4, x:x + 4]
    net = _rrm().net_from_specs([sp], n=2)
    net.set_options(chunk_dense_activity=0.1, stack_dense_activity=2.0)
    net.keyframe(_frame_to_dev([sp], video[0]))
    variants, keep = [], []
    for k in range(3):
        frames = torch.stack([_frame_to_dev([sp], f) for f in video[1 + k * T:1 + (k + 1) * T]])
        outs = net.new_output(frames=T)
        keep.append((frames, outs))
        net.step_seq(frames, outs, T)
        variants.append(net.stats(0)["variant"])              # synchronises: the next call sees this chunk's activity
        for i in (0, T - 1):
            want = orc.dense_forward([sp], video[1 + k * T + i])[0][1]
            got = outs[i].cpu().numpy()
            if dtype == "f32":
                assert float(np.abs(got - want).max()) <= F32_TOL * float(np.abs(want).max()), (k, i)
            else:
                np.testing.assert_array_equal(got.astype(np.int64), want, err_msg=f"chunk {k} frame {i}")
        _compare([sp], net, video[(k + 1) * T], (k + 1) * T)
    assert (variants[1] == 3) == (T >= 8), variants
    net.close()


def test_layers_dense_inside_delta_chunks_count_their_accumulator_tiles():
    """A layer that the per-layer choice evaluates densely inside delta chunks still reports how many accumulator tiles its
    update would touch, so that a chunk in which everything changes lets the next one go dense as a whole."""
    rng = np.random.default_rng(77)
    T, sp = 8, _spec("i8", 40, (64, 64), 36, 3, 1, 1, rng)
    video = np.empty((1 + 3 * T, 1, 40, 64, 64), np.int8)
    video[0] = rng.integers(0, 128, size=video[0].shape)
    for t in range(1, 1 + T):                                 # an eighth of the rows changes: enough for the layer, too little for the chunk
        video[t] = video[t - 1]
        video[t, :, :, :8] = 127 - video[t - 1, :, :, :8]
    for t in range(1 + T, 1 + 3 * T):
        video[t] = 127 - video[t - 1]
    net = _rrm().net_from_specs([sp])
    net.set_options(layer_dense_activity=0.1, layer_delta_activity=0.05, chunk_dense_activity=0.5, stack_dense_activity=2.0)
    net.keyframe(dev(video[0]))
    outs, seen = net.new_output(frames=T), []
    for k in range(3):
        net.step_seq(dev(video[1 + k * T:1 + (k + 1) * T]), outs, T)
        st = net.stats(0)                                     # synchronises: the next call sees this chunk's counters
        seen.append((st["variant"], st["nnz_elems"] >= 0))
        for i in (0, T - 1):
            want = orc.dense_forward([sp], video[1 + k * T + i])[0][1]
            np.testing.assert_array_equal(outs[i].cpu().numpy().astype(np.int64), want, err_msg=f"chunk {k} frame {i}")
    # sparse; dense inside the delta step, counted; dense as a whole, nothing counted
    assert seen == [(2, True), (3, True), (3, False)], seen
    net.close()


def test_chunks_that_never_go_dense_take_no_memory_for_it():
    """The frame-batched dense form of long chunks is set up once the measured activity asks for it, not with the first
    delta chunk."""
    rng = np.random.default_rng(78)
    T, sp = 16, _spec("i8", 64, (120, 120), 64, 3, 1, 1, rng)
    still = rng.integers(0, 128, size=(1, 1, 64, 120, 120)).astype(np.int8).repeat(1 + T, 0)
    frames = dev(still)
    busy = frames.clone()
    busy[1::2] = 127 - busy[1::2]

    def taken(threshold, *chunks):
        net = _rrm().net_from_specs([sp])
        net.set_options(chunk_dense_activity=threshold, stack_dense_activity=2.0)
        outs = net.new_output(frames=T)
        net.keyframe(frames[0])
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        for c in chunks:
            net.step_seq(c[1:], outs, T)
            torch.cuda.synchronize()
        after = torch.cuda.mem_get_info()[0]
        variant = net.stats(0)["variant"]
        net.close()
        return before - after, variant

    batch = T * 120 * 120 * 64 * 2                            # the batched input and output tensors, at least
    never, v0 = taken(2.0, frames, frames)
    quiet, v1 = taken(0.4, frames, frames)
    dense, v2 = taken(0.4, busy, busy)
    assert (v0, v1, v2) == (2, 2, 3)
    assert abs(quiet - never) < batch // 4 and dense - never >= batch // 2, (never, quiet, dense, batch)


@pytest.mark.parametrize("shift", [0, 7])
def test_dense_chunks_whose_outputs_overlap_their_frames(shift):
    """40 frames go in two parts; the first part's outputs lie on frames of the second."""
    rng = np.random.default_rng(79)
    T, sp = 40, _spec("i8", 64, (9, 10), 64, 3, 1, 1, rng, act="relu", shift=9)
    video = rng.integers(0, 128, size=(T, 1, 64, 9, 10)).astype(np.int8)
    net = _rrm().net_from_specs([sp])
    both = torch.zeros((T + shift, 1, 64, 9, 10), dtype=torch.int8, device="cuda")
    for _ in range(2):
        both[:T] = dev(video)
        net.dense_seq(both[:T], both[shift:], T)
        got = both[shift:].cpu().numpy()
        for t in range(T):
            np.testing.assert_array_equal(got[t].astype(np.int64), orc.dense_forward([sp], video[t])[0][1], err_msg=f"frame {t}")
    net.close()


@pytest.mark.parametrize("threshold,goes", [(0.3, True), (0.8, True), (1.0, True), (1.01, False)])
def test_fp32_chunks_with_everything_changing_go_dense_up_to_a_threshold_of_one(threshold, goes):
    rng = np.random.default_rng(80)
    T, sp = 8, _spec("f32", 20, (24, 23), 24, 3, 1, 1, rng)
    video = rng.standard_normal((2 * T, 1, 20, 24, 23)).astype(np.float32)
    net = _rrm().net_from_specs([sp])
    net.set_options(chunk_dense_activity=threshold, stack_dense_activity=2.0)
    outs = net.new_output(frames=T)
    for k in range(2):
        net.step_seq(dev(video[k * T:(k + 1) * T]), outs, T)
        variant = net.stats(0)["variant"]                     # synchronises: the next call sees this chunk's counters
        _compare([sp], net, video[(k + 1) * T - 1], k)
    assert (variant == 3) == goes, variant
    net.close()


def test_dense_chunks_longer_than_one_batch():
    """Dense chunks are batched over their frames, 32 at most per launch: a chunk of 40 frames of two streams goes in
    two parts.  rrm_net_dense_seq leaves the state alone; a chunk that the density switch evaluates densely leaves
    the state at its last frame."""
    rrm = _rrm()
    specs = wl.alexnet_convs("i8", hw=67, scale=8)
    video = wl.moving_rect_video(frames=81, hw=67, dtype="i8", seed=47, n=2, side=(8, 16))
    net = rrm.net_from_specs(specs, n=2)
    frames = dev(np.ascontiguousarray(video))
    out = net.new_output()
    net.keyframe(frames[0], out)
    outs = net.new_output(frames=40)
    net.dense_seq(frames[1:41], outs, 40)
    for i in (0, 19, 20, 39):
        want = orc.dense_forward(specs, video[1 + i])[0][len(specs)]
        np.testing.assert_array_equal(outs[i].cpu().numpy().astype(np.int64), want, err_msg=f"frame {1 + i}")
    _compare(specs, net, video[0], 0)                       # the state is still the keyframe's
    net.set_options(chunk_dense_activity=0.0)               # every measured activity sends the next chunk to the dense evaluation
    net.step_seq(frames[1:41], outs, 40)                    # (nothing measured yet: the delta path)
    assert net.stats(1)["variant"] != 3
    _compare(specs, net, video[40], 40)
    net.step_seq(frames[41:81], outs, 40)
    assert net.stats(1)["variant"] == 3
    for i in (0, 21, 39):
        want = orc.dense_forward(specs, video[41 + i])[0][len(specs)]
        np.testing.assert_array_equal(outs[i].cpu().numpy().astype(np.int64), want, err_msg=f"frame {41 + i}")
    _compare(specs, net, video[80], 80)
    net.close()


def test_stack_chunks_through_the_pipelined_host_entry_point():
    """Host buffers in, host buffers out, calls queued without waiting: a stack's chunks through
    rrm_net_step_seq_host_async deliver every frame's output."""
    rrm = _rrm()
    specs = wl.alexnet_convs("i8", hw=99, scale=8)
    video = wl.moving_rect_video(frames=12, hw=99, dtype="i8", seed=23, n=1, side=(12, 24))
    net = rrm.net_from_specs(specs, n=1)
    ins = [torch.from_numpy(np.ascontiguousarray(video[a:a + 4])).pin_memory() for a in (0, 4, 8)]
    shape = tuple(net.new_output(frames=4).shape)
    outs = [torch.empty(shape, dtype=torch.int8).pin_memory() for _ in range(3)]
    for x, y in zip(ins, outs):
        net.step_seq_host_async(x, y, 4)
    net.host_sync()
    for k, y in enumerate(outs):
        for i in range(4):
            want = orc.dense_forward(specs, video[4 * k + i])[0][len(specs)]
            np.testing.assert_array_equal(y[i].numpy().astype(np.int64), want, err_msg=f"frame {4 * k + i}")
    net.close()


def test_stack_chunk_longer_than_the_arenas_held():
    """More frames in one call than there are per-frame arenas: arenas are reused, each cleared by the frame that
    takes it over; outputs and state are unchanged."""
    rrm = _rrm()
    specs = wl.alexnet_convs("i8", hw=67, scale=8)
    video = wl.moving_rect_video(frames=71, hw=67, dtype="i8", seed=29, n=1, side=(8, 16))
    net = rrm.net_from_specs(specs, n=1)
    rec = orc.Recurrence(specs, n=1)
    rec.step(np.full_like(video[0], 0))
    frames = dev(np.ascontiguousarray(video))
    outs = net.new_output(frames=70)
    net.step_seq(frames[:70], outs, 70)
    for t in range(70):
        rec.step(video[t])
        if t in (0, 1, 33, 64, 65, 69):
            want = orc.dense_forward(specs, video[t])[0][len(specs)]
            np.testing.assert_array_equal(outs[t].cpu().numpy().astype(np.int64), want, err_msg=f"frame {t}")
    _compare(specs, net, video[69], 69)
    for l in range(len(specs)):
        st = net.stats(l)
        assert st["error_word"] == 0 and st["nnz_elems"] == rec.nnz[l] and st["active_macs"] == rec.macs[l], (l, st)
    out = net.new_output()
    net.step(dev(video[70]), out)
    _compare(specs, net, video[70], 70)
    net.close()


# ------------------------------------------------------------------ explicit batch normalisation as part of f (Sec. 4.5)
@pytest.mark.parametrize("name", ["alex_f32", "resnet_i8", "vgg_i8"])
def test_explicit_bn_stacks_every_frame(name):
    """Stacks whose layers keep their batch normalisation explicit (per-channel affine before requantisation /
    activation / pooling): projections, tensors and counters against the oracle at every frame, a keyframe in between."""
    if name == "alex_f32":
        specs, dt, hw, n = wl.alexnet_convs("f32", hw=99, scale=8), "f32", 99, 1
    elif name == "resnet_i8":
        specs, dt, hw, n = wl.resnet18_convs(hw=96, scale=8), "i8", 96, 2
    else:
        specs, dt, hw, n = wl.vgg16_convs("i8", hw=64, scale=8), "i8", 64, 1
    wl.with_explicit_bn(specs)
    assert all(s.bn_scale is not None for s in specs)
    video = wl.moving_rect_video(frames=6, hw=hw, dtype=dt, seed=29, n=n, side=(10, 20))
    _run(specs, video, n=n, stats=True, keyframe_at=(3,))


@pytest.mark.parametrize("by_layer", [False, True])
@pytest.mark.parametrize("name", ["alex_f32", "resnet_i8"])
def test_explicit_bn_stacks_in_chunks(name, by_layer, monkeypatch):
    """The same stacks through rrm_net_step_seq, frame-pipelined and layer by layer over all frames of a chunk:
    every frame's output, then projections and tensors after the chunk."""
    if by_layer:
        monkeypatch.setenv("RRM_CHUNK_BY_LAYER", "1")
    rrm = _rrm()
    if name == "alex_f32":
        specs, dt, hw, n = wl.alexnet_convs("f32", hw=99, scale=8), "f32", 99, 1
    else:
        specs, dt, hw, n = wl.resnet18_convs(hw=96, scale=8), "i8", 96, 2
    wl.with_explicit_bn(specs)
    video = wl.moving_rect_video(frames=9, hw=hw, dtype=dt, seed=37, n=n, side=(10, 20))
    net = rrm.net_from_specs(specs, n=n)
    frames = dev(np.ascontiguousarray(video))
    t0 = 0
    for T in (5, 4):
        outs = net.new_output(frames=T)
        net.step_seq(frames[t0:t0 + T], outs, T)
        for i in range(T):
            want = orc.dense_forward(specs, video[t0 + i])[0][len(specs)]
            got = outs[i].cpu().numpy()
            if dt == "f32":
                assert float(np.abs(got - want).max()) <= F32_TOL * max(1e-30, float(np.abs(want).max())), t0 + i
            else:
                np.testing.assert_array_equal(got.astype(np.int64), want, err_msg=f"frame {t0 + i}")
        t0 += T
        _compare(specs, net, video[t0 - 1], t0 - 1)
    for l in range(len(specs)):
        assert net.stats(l)["error_word"] == 0
    net.close()


def test_explicit_bn_equals_the_folded_stack_on_the_gpu():
    """fp32: the stack with its affines unfolded and the stack with them folded into filters and bias give the same
    tensors within the fp32 tolerance, on the library's delta path."""
    rrm = _rrm()
    specs = wl.with_explicit_bn(wl.alexnet_convs("f32", hw=99, scale=8))
    folded = wl.fold_bn_f32(specs)
    video = wl.moving_rect_video(frames=5, hw=99, dtype="f32", seed=30, side=(10, 20))
    a, b = rrm.net_from_specs(specs), rrm.net_from_specs(folded)
    oa, ob = a.new_output(), b.new_output()
    for t in range(5):
        a.step(dev(video[t]), oa)
        b.step(dev(video[t]), ob)
        scale = float(ob.abs().max())
        assert float((oa - ob).abs().max()) <= 5 * F32_TOL * max(scale, 1e-6), t
    # removing the affine again gives the plain stack's fresh state
    plain = wl.alexnet_convs("f32", hw=99, scale=8)
    for l in range(len(specs)):
        a.set_affine(l, None, None)
    a.step(dev(video[0]), oa)
    want = orc.dense_forward(plain, video[0])[0][len(plain)]
    assert float(np.abs(oa.cpu().numpy() - want).max()) <= F32_TOL * float(np.abs(want).max())
    a.close(); b.close()


def test_affine_is_rejected_where_it_is_not_defined():
    rrm = _rrm()
    specs = wl.xnor_alexnet_convs(hw=99, scale=8)
    net = rrm.net_from_specs(specs)
    z = torch.zeros(specs[0].c_out, dtype=torch.int32, device="cuda")
    with pytest.raises(rrm.RRMError):
        net.set_affine(0, z, z)               # a sign layer
    with pytest.raises(rrm.RRMError):
        net.set_affine(0, z, None)
    net.close()


# ------------------------------------------------------------------ fp32 results are reproducible bit for bit
@pytest.mark.parametrize("name", ["cfg1", "alex_f32"])
def test_fp32_projections_are_bitwise_reproducible(name):
    """Layers whose K range is split over CTAs add their shares' partial sums in a fixed order, so two runs over the
    same frames leave bit-identical projections (the race detector of last resort: any unordered float addition or
    data race would show here)."""
    rrm = _rrm()
    if name == "cfg1":
        specs, video = wl.single_conv_f32(), wl.block_redraw_sequence()
    else:
        specs, video = wl.alexnet_convs("f32", hw=131, scale=4), wl.moving_rect_video(frames=6, hw=131, dtype="f32", seed=3, side=(12, 24))
    runs = []
    for rep in range(3):
        net = rrm.net_from_specs(specs, variant="tensor")      # (no density switch: every frame through the delta kernels)
        out = net.new_output()
        for t in range(video.shape[0]):
            net.step(dev(video[t]), out)
        runs.append([net.projection(l).clone() for l in range(len(specs))] + [out.clone()])
        net.close()
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert torch.equal(a, b)


@pytest.mark.parametrize("how", ["variant", "options", "waits"])
def test_fp32_chunks_are_bitwise_reproducible(how):
    """Delta and dense forms of an fp32 chunk round differently, and which one runs depends on whether the counters of the
    chunk before have arrived.  With the variant pinned, with the thresholds out of reach, or with a wait for each chunk
    before the next, the same video gives the same bits."""
    rrm = _rrm()
    specs, T = wl.alexnet_convs("f32", hw=131, scale=4), 8
    video = dev(np.ascontiguousarray(wl.moving_rect_video(frames=1 + 4 * T, hw=131, dtype="f32", seed=3, side=(12, 24), bg_redraw=0.10)))
    runs, forms = [], []
    for rep in range(3):
        net = rrm.net_from_specs(specs, variant="tensor" if how == "variant" else "auto")
        if how == "options":
            net.set_options(chunk_dense_activity=2.0, stack_dense_activity=2.0)
        net.keyframe(video[0])
        outs, seen = net.new_output(frames=4 * T), []
        for k in range(4):
            net.step_seq(video[1 + k * T:1 + (k + 1) * T], outs[k * T:(k + 1) * T], T)
            if how == "waits":
                torch.cuda.synchronize()
                seen.append(net.stats(1)["variant"])
        runs.append([outs] + [net.projection(l) for l in range(len(specs))])
        forms.append(seen)
        net.close()
    assert forms[0] == forms[1] == forms[2] and (how != "waits" or 3 in forms[0]), forms
    for other in runs[1:]:
        for a, b in zip(runs[0], other):
            assert torch.equal(a, b)


# ------------------------------------------------------------------ chunk forms: layer by layer, frame-pipelined, in place
def _two_layer_stack(dtype, rng):
    """Layer 0 reads a multi-channel input of the given type (the import kernels of every input layout) and pools with
    a window that leaves trailing projection rows outside every window; layer 1 reads its output."""
    if dtype == "bin":
        a = _spec("bin", 40, (15, 14), 36, 3, 1, 1, rng, act="sign", pool=(3, 2, 0), theta=2)
        b = _spec("bin", 36, (7, 6), 20, 3, 1, 1, rng, act="sign", theta=1)
    elif dtype == "i8":
        a = _spec("i8", 16, (16, 14), 40, 3, 1, 1, rng, act="relu", pool=(3, 2, 0), shift=11)
        b = _spec("i8", 40, (7, 6), 24, 3, 1, 1, rng, act="none")
    else:
        a = _spec("f32", 12, (16, 14), 40, 3, 1, 1, rng, act="relu", pool=(2, 2, 0))
        b = _spec("f32", 40, (8, 7), 24, 3, 1, 1, rng, act="leaky")
    b.src = 1
    return [a, b]


@pytest.mark.parametrize("form", ["layer_by_layer", "pipelined", "in_place"])
@pytest.mark.parametrize("dtype", ["f32", "i8", "bin"])
def test_chunk_forms_agree_with_the_oracle(dtype, form, monkeypatch):
    """rrm_net_step_seq on a delta chunk has three forms (every kernel over all frames of the chunk; frames
    overlapping in one graph with the frame's product kept apart; the same adding in place).  Each must give every
    frame's output, the state after the chunk and the last frame's counters of Algorithm 1 - also across a frame
    without change and a frame in which everything changes, for every input layout, two streams."""
    if form == "layer_by_layer":
        monkeypatch.setenv("RRM_CHUNK_BY_LAYER", "1")
    elif form == "pipelined":
        monkeypatch.setenv("RRM_CHUNK_PIPELINED", "1")
    elif form == "in_place":
        monkeypatch.setenv("RRM_CHUNK_INPLACE", "1")
    rrm = _rrm()
    rng = np.random.default_rng({"f32": 5, "i8": 6, "bin": 7}[dtype])
    specs = _two_layer_stack(dtype, rng)
    s0 = specs[0]
    video = _video(dtype, s0.c_in, (s0.h, s0.w), 10, 2, rng)
    net = rrm.net_from_specs(specs, n=2)
    rec = orc.Recurrence(specs, n=2)
    rec.step(np.full_like(video[0], -1 if dtype == "bin" else 0))
    packed = [_frame_to_dev(specs, video[t]) for t in range(video.shape[0])]
    t0 = 0
    for T in (4, 3, 2):
        frames = torch.stack(packed[t0:t0 + T]).contiguous()
        outs = net.new_output(frames=T)
        net.step_seq(frames, outs, T)
        for i in range(T):
            rec.step(video[t0 + i])
            want = orc.dense_forward(specs, video[t0 + i])[0][len(specs)]
            got = outs[i].cpu().numpy()
            if dtype == "f32":
                assert float(np.abs(got - want).max()) <= F32_TOL * max(1e-30, float(np.abs(want).max())), t0 + i
            elif dtype == "bin":
                np.testing.assert_array_equal(unpack_bits_nhwc(got.view(np.uint32), specs[-1].c_out), want, err_msg=f"frame {t0 + i}")
            else:
                np.testing.assert_array_equal(got.astype(np.int64), want, err_msg=f"frame {t0 + i}")
        t0 += T
        _compare(specs, net, video[t0 - 1], t0 - 1)
        for l in range(len(specs)):
            st = net.stats(l)
            assert st["error_word"] == 0
            if dtype != "f32" or l == 0:
                assert st["nnz_elems"] == rec.nnz[l] and st["active_macs"] == rec.macs[l], (form, t0, l, st, rec.nnz[l], rec.macs[l])
    out = net.new_output()
    net.step(packed[9], out)                  # a single step carries on from the chunk's state
    _compare(specs, net, video[9], 9)
    net.close()
