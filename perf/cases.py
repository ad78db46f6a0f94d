"""What a user of this library has it do, as timed cases: video frames through residual layers and stacks.

A case is one network (a lone fully connected layer, a lone convolution, or a stack shaped like AlexNet, ResNet-18 or the
XNOR AlexNet), a number of independent video streams per call, and a call:

    call "delta", frames 1     one frame of every stream          (Net.step)
    call "delta", frames > 1   a chunk of consecutive frames      (Net.step_seq)
    call "dense", frames 1     a keyframe that resets the state   (Net.keyframe)
    call "dense", frames > 1   frames evaluated on their own      (Net.dense_seq)

Every pass takes the next frame (or chunk) of a video that is under way: prepare() leaves a net whose keyframe and first
pass lie behind it, and the passes walk the video forwards and backwards, so that no pass repeats its predecessor's
frame.  All inputs are drawn from the seed, on the GPU."""
import math
import random

import torch

import paper_1802_09723_b200 as rrm

STEP_FRAMES = 9          # frames of the video that a case of one frame per call walks over


# ------------------------------------------------------------------------------------------------ networks
class Spec:
    """One linear layer and the map after it, with the attributes rrm.desc_from_spec reads."""

    def __init__(self, kind, dtype, c_in, hw, c_out, k=1, stride=1, pad=0, act="relu", pool=None, shift=0, src=-1, res=-1):
        self.kind, self.dtype, self.c_in, self.h, self.w, self.c_out = kind, dtype, c_in, hw, hw, c_out
        self.kh = self.kw = k
        self.stride, self.pad, self.act, self.pool, self.theta = stride, pad, act, pool, 0
        self.shift, self.src, self.res = (-1 if dtype == "f32" else shift), src, res

    @property
    def p_hw(self):
        return (self.h + 2 * self.pad - self.kh) // self.stride + 1

    @property
    def out_hw(self):
        if self.pool is None:
            return self.p_hw
        k, s, p = self.pool
        return (self.p_hw + 2 * p - k) // s + 1

    @property
    def macs(self):
        return self.p_hw ** 2 * self.c_out * self.c_in * self.kh * self.kw


def alexnet(dtype, hw):
    """conv1 .. conv5, fp32 or int8; "bin": conv1 int8, the others +-1 weights and inputs, as in an XNOR network."""
    plan = ((96, 11, 4, 0, True), (256, 5, 1, 2, True), (384, 3, 1, 1, False), (384, 3, 1, 1, False), (256, 3, 1, 1, True))
    layers, c, size = [], 3, hw
    for i, (c_out, k, stride, pad, pooled) in enumerate(plan):
        act = "relu" if dtype != "bin" else ("sign" if i < 4 else "none")
        layers.append(Spec("conv", "i8" if dtype == "bin" and i == 0 else dtype, c, size, c_out, k, stride, pad, act,
                           (3, 2, 0) if pooled else None, -1 if dtype == "bin" else 0, src=i))
        c, size = c_out, layers[-1].out_hw
    return layers


def resnet18(hw):
    """The 20 convolutions of ResNet-18, int8, with identity and 1x1 stride-2 shortcuts."""
    layers = [Spec("conv", "i8", 3, hw, 64, 7, 2, 3, "relu", (3, 2, 1), src=0)]
    tensor, c, size = 1, 64, layers[0].out_hw
    for stage, width in enumerate((64, 128, 256, 512)):
        for block in range(2):
            stride = 2 if stage > 0 and block == 0 else 1
            layers.append(Spec("conv", "i8", c, size, width, 3, stride, 1, src=tensor))
            mid, shortcut = len(layers), tensor
            if stride != 1 or c != width:
                layers.append(Spec("conv", "i8", c, size, width, 1, stride, 0, "none", src=tensor))
                shortcut = len(layers)
            layers.append(Spec("conv", "i8", width, layers[mid - 1].out_hw, width, 3, 1, 1, src=mid, res=shortcut))
            tensor, c, size = len(layers), width, layers[-1].out_hw
    return layers


def network(case):
    net, dtype = case["net"], case["dtype"]
    if net == "fc":
        return [Spec("fc", "i8", case["c_in"], 1, case["c_out"], act="none", shift=-1, src=0)]
    if net == "layer":
        k = case["k"]
        act = "none" if dtype == "f32" else "relu"
        return [Spec("conv", dtype, case["c_in"], case["hw"], case["c_out"], k, 1, k // 2, act, src=0)]
    return resnet18(case["hw"]) if net == "resnet18" else alexnet(dtype, case["hw"])


def fill(layers, g):
    """Random weights and biases (He-init; int8 scaled to +-127), with the requantisation shift and the sign threshold
    that their statistics call for, so that activations neither die nor saturate."""
    weights, biases = [], []
    for s in layers:
        shape, fan_in = (s.c_out, s.c_in, s.kh, s.kw), s.c_in * s.kh * s.kw
        if s.kind == "fc":
            weights.append(torch.randint(-127, 128, shape, dtype=torch.int8, device="cuda", generator=g))
            biases.append(torch.randint(-1000, 1001, (s.c_out,), dtype=torch.int32, device="cuda", generator=g))
            continue
        w = torch.randn(shape, device="cuda", generator=g)
        if s.dtype == "f32":
            weights.append(w * math.sqrt(2.0 / fan_in))
            biases.append(torch.randn(s.c_out, device="cuda", generator=g) * 0.1)
            continue
        q = torch.where(w >= 0, 1, -1).to(torch.int8) if s.dtype == "bin" else (w / w.abs().max() * 127).round().to(torch.int8)
        spread = math.sqrt(fan_in * float(q.double().square().mean()))
        sigma = spread * (1.0 if s.dtype == "bin" else 37.0 if s.src == 0 else 32.0)
        noise = max(1, int(sigma / 8))
        b = torch.randint(-noise, noise + 1, (s.c_out,), device="cuda", generator=g)
        if s.dtype == "i8" and s.src == 0:              # pixels in [0, 127]: centre them
            b = b - 64 * q.long().sum(dim=(1, 2, 3))
        if s.shift >= 0:
            s.shift = max(0, round(math.log2(spread)))
        if s.act == "sign" and s.pool is not None:      # (a maximum over a window lies above the median)
            s.theta = round(sigma)
        weights.append(q)
        biases.append(b.to(torch.int32))
    return weights, biases


# ------------------------------------------------------------------------------------------------ inputs
def pixels(shape, dtype, g):
    if dtype == "f32":
        return torch.rand(shape, device="cuda", generator=g)
    return torch.randint(0, 128, shape, dtype=torch.int8, device="cuda", generator=g)


def fc_sequence(case, frames, g):
    """Feature vectors in which runs of 32 entries, `rho` of all, take new values from frame to frame."""
    n, c = case["streams"], case["c_in"]
    slots = c // 32
    out = torch.empty((frames, n, c), dtype=torch.int8, device="cuda")
    out[0] = pixels((n, c), "i8", g)
    for t in range(1, frames):
        out[t] = out[t - 1]
        pick = torch.rand((n, slots), device="cuda", generator=g).topk(max(1, round(case["rho"] * slots))).indices
        mask = torch.zeros((n, slots), dtype=torch.bool, device="cuda").scatter_(1, pick, True).repeat_interleave(32, 1)
        mask = torch.nn.functional.pad(mask, (0, c - 32 * slots)).roll(5 * t, 1)
        out[t] = torch.where(mask, pixels((n, c), "i8", g), out[t])
    return out


def patch_sequence(case, frames, g, r):
    """Feature maps (after a ReLU) in which 8 x 8 patches, a tenth of the area, take new values from frame to frame."""
    n, c, hw = case["streams"], case["c_in"], case["hw"]

    def draw():
        return torch.randn((n, c, hw, hw), device="cuda", generator=g).clamp_min_(0) if case["dtype"] == "f32" else pixels((n, c, hw, hw), "i8", g)

    out = torch.empty((frames, n, c, hw, hw), dtype=torch.float32 if case["dtype"] == "f32" else torch.int8, device="cuda")
    out[0] = draw()
    for t in range(1, frames):
        mask = torch.zeros((n, 1, hw, hw), dtype=torch.bool)
        for s in range(n):
            for _ in range(math.ceil(0.10 * hw * hw / 64)):
                y, x = r.randrange(hw - 7), r.randrange(hw - 7)
                mask[s, :, y:y + 8, x:x + 8] = True
        out[t] = torch.where(mask.cuda(), draw(), out[t - 1])
    return out


def video(case, frames, g, r):
    """Textured rectangles that move over a still background and bounce off its edges.  "busy": three of 32-64 pixels,
    1-4 pixels a frame; "quiet": one of 24-32, 1-2 pixels a frame; "noisy": busy, and a fiftieth of the background
    pixels takes new values in every frame."""
    n, hw, dtype, motion = case["streams"], case["hw"], "f32" if case["dtype"] == "f32" else "i8", case["motion"]
    back = pixels((n, 3, hw, hw), dtype, g)
    out = torch.empty((frames, n, 3, hw, hw), dtype=back.dtype, device="cuda")
    side, speed, count = ((24, 32), (1, 2), 1) if motion == "quiet" else ((32, 64), (1, 4), 3)
    rects = []
    for s in range(n):
        for _ in range(count):
            h, w = r.randint(*side), r.randint(*side)
            rects.append([s, h, w, pixels((3, h, w), dtype, g), r.randint(0, hw - h), r.randint(0, hw - w),
                          r.choice((-1, 1)) * r.randint(*speed), r.choice((-1, 1)) * r.randint(*speed)])
    for t in range(frames):
        if t and motion == "noisy":
            mask = torch.rand((n, 1, hw, hw), device="cuda", generator=g) < 0.02
            back = torch.where(mask, pixels((n, 3, hw, hw), dtype, g), back)
        out[t] = back
        for q in rects:
            s, h, w, texture, y, x, vy, vx = q
            if t:
                y, x = y + vy, x + vx
                if not 0 <= y <= hw - h:
                    y, vy = (-y if y < 0 else 2 * (hw - h) - y), -vy
                if not 0 <= x <= hw - w:
                    x, vx = (-x if x < 0 else 2 * (hw - w) - x), -vx
                q[4:] = y, x, vy, vx
            out[t, s, :, y:y + h, x:x + w] = texture
    return out


# ------------------------------------------------------------------------------------------------ the cases
def listed():
    fc = {"net": "fc", "dtype": "i8", "call": "delta"}
    return [
        # the smallest call: one feature vector of one stream through a 9216 -> 4096 layer, frame by frame as it arrives
        dict(fc, name="fc_frame", streams=1, frames=1, c_in=9216, c_out=4096, rho=0.05),
        # the same layer fed with a recorded video, 32 frames per call (the benchmark's workload)
        dict(fc, name="fc_chunk", streams=1, frames=32, c_in=9216, c_out=4096, rho=0.05),
        # a server that steps 11 cameras together through a classifier layer, a few frames at a time
        dict(fc, name="fc_streams", streams=11, frames=5, c_in=4096, c_out=1008, rho=0.02),
        # one fp32 convolution inside somebody else's network, frame by frame
        {"name": "layer_f32_frame", "net": "layer", "dtype": "f32", "call": "delta", "streams": 1, "frames": 1, "c_in": 64, "c_out": 64, "k": 3, "hw": 56},
        # an int8 convolution of uneven sizes, three streams, chunks of ten frames
        {"name": "layer_i8_chunk", "net": "layer", "dtype": "i8", "call": "delta", "streams": 3, "frames": 10, "c_in": 48, "c_out": 80, "k": 5, "hw": 45},
        # an fp32 network over eight cameras, one frame of each per call
        {"name": "alexnet_f32_streams", "net": "alexnet", "dtype": "f32", "call": "delta", "streams": 8, "frames": 1, "hw": 227, "motion": "busy"},
        # the same network over a recorded video
        {"name": "alexnet_f32_chunk", "net": "alexnet", "dtype": "f32", "call": "delta", "streams": 1, "frames": 32, "hw": 227, "motion": "busy"},
        # the quantised network on one camera, where the time until the answer counts
        {"name": "alexnet_i8_frame", "net": "alexnet", "dtype": "i8", "call": "delta", "streams": 1, "frames": 1, "hw": 227, "motion": "busy"},
        # the quantised network over a recorded video
        {"name": "alexnet_i8_chunk", "net": "alexnet", "dtype": "i8", "call": "delta", "streams": 1, "frames": 32, "hw": 227, "motion": "busy"},
        # keyframes of many streams at once: precise inference, at a size that is no multiple of anything
        {"name": "alexnet_i8_keyframe", "net": "alexnet", "dtype": "i8", "call": "dense", "streams": 24, "frames": 1, "hw": 195, "motion": "busy"},
        # a binary network watching quiet scenes, two streams, chunks of 25 frames
        {"name": "xnor_chunk", "net": "alexnet", "dtype": "bin", "call": "delta", "streams": 2, "frames": 25, "hw": 227, "motion": "quiet"},
        # a residual network on four cameras with sensor noise, frame by frame
        {"name": "resnet18_i8_streams", "net": "resnet18", "dtype": "i8", "call": "delta", "streams": 4, "frames": 1, "hw": 224, "motion": "noisy"},
    ]


def _spread(rng, lo, hi):
    """A whole number whose logarithm is uniform."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    kind = rng.choice(("fc", "layer", "alexnet", "alexnet", "alexnet", "resnet18"))
    call = "delta" if rng.random() < 0.75 else "dense"
    if kind == "fc":
        return {"net": "fc", "dtype": "i8", "call": call, "streams": _spread(rng, 1, 16), "frames": _spread(rng, 1, 32),
                "c_in": 16 * _spread(rng, 40, 576), "c_out": 16 * _spread(rng, 16, 256), "rho": round(_spread(rng, 10, 200) / 1000, 3)}
    if kind == "layer":
        case = {"net": "layer", "dtype": rng.choice(("f32", "i8")), "call": call, "streams": 1, "frames": 1, "c_in": rng.randint(16, 128),
                "c_out": rng.randint(16, 128), "k": rng.choice((1, 3, 5)), "hw": rng.randint(28, 90)}
    elif kind == "alexnet":
        case = {"net": "alexnet", "dtype": rng.choice(("f32", "i8", "bin")), "call": call, "streams": 1, "frames": 1,
                "hw": rng.randint(131, 227), "motion": rng.choice(("busy", "quiet", "noisy"))}
    else:
        case = {"net": "resnet18", "dtype": "i8", "call": call, "streams": 1, "frames": 1, "hw": rng.randint(131, 224),
                "motion": rng.choice(("busy", "quiet", "noisy"))}
    # as many frames and streams as keep the pass at most as large as the fp32 chunk of listed(): 32 frames of 1.07 GMAC
    most = min(256, int(34e9 / sum(s.macs for s in network(case))))
    case["streams"] = _spread(rng, 1, min(32, most))
    case["frames"] = _spread(rng, 1, max(1, min(32, most // case["streams"])))
    return case


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = random.Random(seed)
    layers = network(case)
    weights, biases = fill(layers, g)
    net = rrm.Net([rrm.desc_from_spec(s, case["streams"]) for s in layers], weights, biases)
    T = case["frames"]
    count = STEP_FRAMES if T == 1 else T + 1
    if case["net"] == "fc":
        seq = fc_sequence(case, count, g)
    elif case["net"] == "layer":
        seq = patch_sequence(case, count, g, r)
    else:
        seq = video(case, count, g, r)
    if T == 1:
        clips = [seq[i] for i in list(range(1, count)) + list(range(count - 2, -1, -1))]
    else:
        clips = [seq[1:], seq[:-1].flip(0).contiguous()]
    state = {"net": net, "seq": seq, "clips": clips, "at": 0, "dense": case["call"] == "dense", "frames": T,
             "out": net.new_output(frames=None if T == 1 else T)}
    net.keyframe(seq[0])
    run(state)                                           # the video is under way
    return state


def run(state):
    net, out = state["net"], state["out"]
    clip = state["clips"][state["at"]]
    state["at"] = (state["at"] + 1) % len(state["clips"])
    if state["frames"] == 1:
        (net.keyframe if state["dense"] else net.step)(clip, out)
    else:
        (net.dense_seq if state["dense"] else net.step_seq)(clip, out)
    return out


# share of a dense pass's multiply-accumulates that the non-zero deltas imply (the library's own counters)
SHARE = {"busy": 0.23, "quiet": 0.05, "noisy": 0.55}


def work(case):
    layers, T, n = network(case), case["frames"], case["streams"]
    delta = case["call"] == "delta"
    size = {"f32": 4, "i8": 1, "bin": 1 / 8}
    first, last = layers[0], layers[-1]
    share = 1.0
    if delta:
        share = case["rho"] if case["net"] == "fc" else 0.10 if case["net"] == "layer" else SHARE[case["motion"]]
    weights = sum(s.c_out * s.c_in * s.kh * s.kw * size[s.dtype] for s in layers)
    if delta and case["net"] == "fc":                    # the columns of the inputs that change in some frame
        weights *= 1 - (1 - share) ** (T * n)
    frames = T * n * first.c_in * first.h * first.w * size[first.dtype]
    outs = T * n * last.c_out * last.out_hw ** 2 * (4 if last.shift < 0 else 1)
    # a delta pass reads its predecessor's projections where they change, and a pass that keeps a state writes it
    held = sum(n * s.c_out * s.p_hw ** 2 * 4 for s in layers) + frames / T
    state = 2 * share * held if delta else (held if T == 1 else 0)
    return {"bytes": weights + frames + outs + state, "flops": 2.0 * share * T * n * sum(s.macs for s in layers)}


def tolerance(case):
    """Integer results are unique.  fp32 sums may be taken in any order: against the same network in 64 bits the fp32 cases
    differ by up to 1.2e-6 (2-norm) and 8.7e-6 (largest) after some forty frames of the recurrence."""
    if case["dtype"] != "f32":
        return "exact"
    return {"rel": 5e-6, "max": 4e-5}
