"""How convolution launches are cut, by host arithmetic (no GPU): every layer that the tensor-core kernel takes has a plan
for every launch it can come to."""
import random

import workloads as wl
import paper_1802_09723_b200 as rrm

FORMS = (("delta", 1), ("pipelined", 1), ("dense", 1), ("dense", 7), ("dense", 32), ("seq", 2), ("seq", 32))


def desc(dtype, c_in, h, w, c_out, kh, kw, stride, pad, n):
    d = rrm.LayerDesc()
    d.kind, d.dtype, d.n, d.c_in, d.h, d.w, d.c_out = 0, rrm.DTYPE[dtype], n, c_in, h, w, c_out
    d.kh, d.kw, d.stride, d.pad, d.shift, d.res = kh, kw, stride, pad, -1, -1
    return d


def test_layers_of_wide_windows_have_a_plan_for_every_launch():
    """First layers whose window leaves room for the filter stages of one tile width only: stages are 12 KB for tiles of 96
    columns and 16 KB for those of 128 and of 32."""
    taken = 0
    for shape in (("i8", 4, 19, 77, 162, 11, 11, 1, 3, 2), ("i8", 3, 64, 1110, 64, 9, 9, 3, 0, 1), ("i8", 3, 64, 1110, 96, 9, 9, 3, 0, 1),
                  ("i8", 4, 31, 87, 96, 11, 11, 1, 5, 1), ("i8", 3, 40, 91, 70, 11, 11, 1, 0, 1)):
        for form, frames in FORMS:
            taken += rrm.plan_conv(desc(*shape), form, frames)["columns"] > 0      # (raises if a launch has no plan)
    assert taken > 0


def test_every_layer_that_is_taken_has_a_plan_for_every_launch():
    r = random.Random(1)
    taken = 0
    for _ in range(6000):
        k = r.randint(1, 11)
        kw = k if r.random() < 0.6 else r.randint(1, min(16, 128 // k))
        dtype = r.choice(("i8", "i8", "i8", "bin", "f32"))
        c_in = r.randint(1, 4) if r.random() < 0.5 else r.randint(5, 300)
        h, w = r.randint(k, 90), r.randint(kw, 1200)
        d = desc(dtype, c_in, h, w, r.randint(1, 512), k, kw, r.randint(1, 4), r.randint(0, min(k, kw) - 1), r.randint(1, 3))
        for form, frames in FORMS:
            try:
                p = rrm.plan_conv(d, form, frames)
            except rrm.RRMError as e:
                assert "(-5)" in str(e), (str(e), form, frames, [getattr(d, f) for f, _ in d._fields_])     # (more than 2^31 elements)
                continue
            taken += p["columns"] > 0
    assert taken > 10000


def test_filters_are_held_as_narrow_tiles_only_where_a_launch_can_take_them():
    """A dense pass takes 32-column tiles while twice the wide tiles (128 pixels x up to 128 channels) fit 148 CTAs; a layer with more
    of them in one frame, of 32 columns anyway, or of floats holds its filters once."""
    for shape, want in ((("i8", 64, 14, 14, 256, 3, 3, 1, 1, 1), 1),
                        (("i8", 64, 96, 97, 64, 3, 3, 1, 1, 1), 1),          # 74 tiles
                        (("i8", 64, 97, 97, 64, 3, 3, 1, 1, 1), 0),          # 75
                        (("bin", 64, 97, 97, 64, 3, 3, 1, 1, 1), 0),
                        (("i8", 64, 56, 56, 256, 3, 3, 1, 1, 24), 0),
                        (("i8", 64, 14, 14, 32, 3, 3, 1, 1, 1), 0), (("f32", 64, 14, 14, 256, 3, 3, 1, 1, 1), 0)):
        d = desc(*shape)
        assert rrm.plan_conv(d, "dense")["narrow_filters"] == want, shape
        for form, frames in FORMS:
            p = rrm.plan_conv(d, form, frames)
            assert want or p["columns"] != 32 or shape[4] <= 32


def test_narrow_tiles_are_taken_where_every_one_lays_out_few_windows():
    """Few blocks of the K loop: 32 columns; many, of several planes or of 1x1 filters: wide tiles whose shares divide them.  The
    same for the deltas whose shares form a cluster (channels that are no multiple of 4)."""
    for shape, form, want in ((("i8", 28, 23, 26, 239, 5, 5, 1, 0, 2), "dense", 32), (("i8", 96, 27, 27, 256, 5, 5, 1, 2, 1), "dense", 32),
                              (("i8", 256, 14, 14, 512, 3, 3, 2, 1, 4), "dense", 32), (("bin", 127, 13, 9, 185, 1, 1, 3, 0, 2), "dense", 32),
                              (("i8", 3, 227, 227, 96, 11, 11, 4, 0, 1), "dense", 32), (("i8", 384, 11, 11, 384, 3, 3, 1, 1, 1), "dense", 32),
                              (("i8", 409, 112, 120, 85, 3, 3, 3, 0, 3), "dense", 96), (("bin", 414, 96, 74, 84, 3, 3, 2, 1, 3), "dense", 96),
                              (("i8", 1024, 14, 14, 256, 1, 1, 1, 0, 2), "dense", 128), (("i8", 455, 47, 30, 57, 3, 3, 2, 1, 8), "dense", 64),
                              (("bin", 272, 67, 103, 481, 3, 3, 2, 1, 1), "delta", 128), (("i8", 104, 8, 11, 170, 3, 3, 1, 0, 11), "delta", 32),
                              (("bin", 59, 50, 46, 91, 3, 3, 2, 0, 12), "delta", 96), (("bin", 59, 50, 46, 91, 3, 3, 2, 0, 12), "dense", 32)):
        p = rrm.plan_conv(desc(*shape), form)
        assert p["columns"] == want and (p["clustered"] or p["shares"] == 1), (shape, p)


def test_layers_of_stacks_are_planned_like_lone_ones():
    for s in wl.resnet18_convs(hw=64):
        d = rrm.desc_from_spec(s, 2)
        assert rrm.plan_conv(d, "dense") == rrm.plan_conv(desc(s.dtype, s.c_in, s.h, s.w, s.c_out, s.kh, s.kw, s.stride, s.pad, 2), "dense")
