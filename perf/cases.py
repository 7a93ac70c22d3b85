"""The convolution calls whose speed is measured, from the smallest single layer to the largest batch.

Every case goes through the package's public calls: a plan that is created once per layer shape (embedding by
timed selection), given its weights and then run on fresh activations; the one-shot call, which takes weights and
activations together; the streaming call on host buffers; and a short stack of layers that hand int8 NHWC
activations to each other.  Shapes are the five benchmark shapes of ``synth.CONFIGS`` at the batch sizes of the
benchmark's contract and scaled series, the shapes of its candidate report, and sizes between them.
"""
import math

import torch

import paper_2104_04731_b200 as b2c

# One dictionary per layer: every field of a convolution, as plain numbers.  stride / pad / dil apply to both axes.
_FIELDS = dict(kind="plan", N=1, C=1, H=1, W=1, K=1, R=1, S=1, stride=1, pad=0, dil=1, shift=0, groups=1,
               in_layout=b2c.LAYOUT_NCHW, out_layout=b2c.LAYOUT_NCHW, out_mode=b2c.OUT_I32, act=0, calls=1)


def _case(name=None, **kw):
    c = dict(_FIELDS)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # One small layer of one image, both outputs: the smallest call, where launches and host work count.
        _case("layer_c16_14x14_n1", N=1, C=16, H=14, W=14, K=16, R=3, S=3, pad=1, shift=8, out_mode=3),
        # One image through the one-shot call, for programs that keep no plan: weights are packed on every call.
        _case("oneshot_c64_56x56_n1", kind="oneshot", N=1, C=64, H=56, W=56, K=64, R=3, S=3, pad=1),
        # First layer of an image network on a small batch: three channels, large strided filter.
        _case("image_c3_224x224_n4", N=4, C=3, H=224, W=224, K=64, R=7, S=7, stride=2, pad=3),
        # The same family in an offline batch whose rows are no multiple of 16 bytes (a generic odd image size).
        _case("image_c3_227x227_n64", N=64, C=3, H=227, W=227, K=64, R=7, S=7, stride=2, pad=3),
        # Speech spectrogram layer, one channel, odd width, tall filter (the layer class with the paper's largest gain).
        _case("speech_c1_700x161_n32", N=32, C=1, H=700, W=161, K=32, R=20, S=5, stride=2),
        # The benchmark's compute-bound layer at its contract batch, int8 result for the next layer.
        _case("strided_c256_14x14_n32", N=32, C=256, H=14, W=14, K=512, R=3, S=3, stride=2, pad=1, shift=10, out_mode=2),
        # The same layer in the scaled series: the largest amount of arithmetic.
        _case("strided_c256_14x14_n1440", N=1440, C=256, H=14, W=14, K=512, R=3, S=3, stride=2, pad=1, shift=10, out_mode=2),
        # A large batch of medium images, int32 result: bound by memory traffic.
        _case("batch_c64_56x56_n315", N=315, C=64, H=56, W=56, K=64, R=3, S=3, pad=1),
        # A very large batch of small images and both outputs.
        _case("batch_c16_14x14_n15501", N=15501, C=16, H=14, W=14, K=16, R=3, S=3, pad=1, shift=8, out_mode=3),
        # Four layers of a quantised network in a row, int8 NHWC between them, bias and ReLU on each.
        _case("stack_c3_224x224_n8", kind="stack", N=8, C=3, H=224, W=224, K=64, shift=10),
        # Depth-wise layer, form chosen by timing.
        _case("depthwise_c256_28x28_n128", N=128, C=256, H=28, W=28, K=256, R=3, S=3, pad=1, groups=256),
        # Batches that start and end in host memory: eight calls of the benchmark's layer in flight, then a wait.
        _case("stream_c256_14x14_n32", kind="stream", N=32, C=256, H=14, W=14, K=512, R=3, S=3, stride=2, pad=1,
              shift=10, out_mode=2, calls=8),
    ]


def _log(rng, lo, hi):
    """An integer between lo and hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _fit_batch(rng, c, top, flops=60e9, nbytes=160e6):
    """Draws the batch: at least 1, at most `top`, and within the given work."""
    c["N"] = 1
    w = work(c)
    most = min(top, flops / max(w["flops"], 1), nbytes / max(w["bytes"], 1))
    c["N"] = _log(rng, 1, max(1, most))
    return c


def draw(rng):
    """One more case of the same ranges."""
    family = rng.choice(["layer", "layer", "batch", "image", "speech", "strided", "oneshot", "stack", "grouped", "dilated",
                         "stream"])
    if family in ("layer", "batch", "oneshot"):
        C, K = _log(rng, 12, 256), _log(rng, 12, 512)
        H, W = _log(rng, 7, 112), _log(rng, 7, 112)
        R = rng.choice([1, 3, 3, 3, 5])
        c = _case(C=C, H=H, W=W, K=K, R=R, S=R, stride=rng.choice([1, 1, 2]), pad=R // 2)
        if family == "oneshot":
            c["kind"] = "oneshot"
            c["out_mode"] = rng.choice([1, 2, 3])
        else:
            c["in_layout"] = rng.choice([b2c.LAYOUT_NCHW, b2c.LAYOUT_NCHW, b2c.LAYOUT_NHWC])
            c["out_layout"] = c["in_layout"]
            c["out_mode"] = rng.choice([1, 2, 3])
            c["act"] = rng.choice([0, 1])
        c["shift"] = 0 if c["out_mode"] == 1 else 7 + int(math.log2(C * R * R) / 2)
        return _fit_batch(rng, c, 8 if family == "layer" else 16384)
    if family == "image":
        R = rng.choice([3, 5, 7, 7])
        c = _case(C=rng.choice([1, 3, 3, 3, 4]), H=_log(rng, 96, 256), W=_log(rng, 96, 256), K=rng.choice([16, 24, 32, 64, 64]),
                  R=R, S=R, stride=rng.choice([1, 2, 2]), pad=R // 2, shift=10, out_mode=rng.choice([1, 1, 2]))
        return _fit_batch(rng, c, 100)
    if family == "speech":
        c = _case(C=1, H=_log(rng, 79, 700), W=_log(rng, 161, 480), K=32, R=rng.choice([5, 9, 20]), S=rng.choice([5, 20, 21]),
                  stride=2)
        return _fit_batch(rng, c, 244)
    if family in ("strided", "stream"):
        c = _case(C=32 * rng.randint(2, 8), H=rng.choice([14, 14, 28]), W=rng.choice([14, 14, 28]), K=64 * rng.randint(1, 8), R=3,
                  S=3, stride=2, pad=1, shift=10, out_mode=2)
        if family == "stream":
            c.update(kind="stream", calls=rng.randint(3, 8))
        return _fit_batch(rng, c, 48 if family == "stream" else 1440)
    if family == "stack":
        size = 8 * rng.randint(12, 32)
        return _fit_batch(rng, _case(kind="stack", C=3, H=size, W=size, K=rng.choice([32, 64]), shift=10), 16)
    if family == "grouped":
        C = 32 * rng.randint(2, 12)
        groups = rng.choice([C, C, C // 2, C // 16])
        c = _case(C=C, H=_log(rng, 14, 56), W=_log(rng, 14, 56), K=C, R=3, S=3, pad=1, groups=groups)
        return _fit_batch(rng, c, 128, nbytes=80e6)
    d = rng.choice([2, 2, 4])
    c = _case(C=_log(rng, 3, 64), H=_log(rng, 48, 96), W=_log(rng, 48, 96), K=rng.choice([16, 32, 64]), R=3, S=3, pad=d, dil=d)
    return _fit_batch(rng, c, 64)


def _layers(case):
    """The layers of a stack: a first layer on NCHW images, then NHWC layers; the last one keeps its int32 sums."""
    K = case["K"]
    nchw, nhwc = b2c.LAYOUT_NCHW, b2c.LAYOUT_NHWC
    geo = [  # C, K, filter, stride, pad, shift, input layout, outputs
        (case["C"], K, 7, 2, 3, case["shift"], nchw, b2c.OUT_I8),
        (K, K, 3, 1, 1, case["shift"] + 1, nhwc, b2c.OUT_I8),
        (K, 2 * K, 3, 2, 1, case["shift"] + 1, nhwc, b2c.OUT_I8),
        (2 * K, 4 * K, 1, 1, 0, 0, nhwc, b2c.OUT_I32),
    ]
    out, H, W = [], case["H"], case["W"]
    for C, k, r, s, p, sh, layout, mode in geo:
        out.append(_case(N=case["N"], C=C, H=H, W=W, K=k, R=r, S=r, stride=s, pad=p, shift=sh, in_layout=layout,
                         out_layout=nhwc, out_mode=mode, act=1))
        H, W = (H + 2 * p - r) // s + 1, (W + 2 * p - r) // s + 1
    return out


def _desc(c):
    return b2c.make_desc(c["N"], c["C"], c["H"], c["W"], c["K"], c["R"], c["S"], c["stride"], c["pad"], c["dil"], c["shift"],
                         c["in_layout"], c["out_layout"], c["out_mode"])


def _out_extent(c):
    span = c["dil"] * (c["R"] - 1) + 1, c["dil"] * (c["S"] - 1) + 1
    return (c["H"] + 2 * c["pad"] - span[0]) // c["stride"] + 1, (c["W"] + 2 * c["pad"] - span[1]) // c["stride"] + 1


_chosen = {}


def _make_plan(c):
    """A plan with the timed embedding.  A program times a layer shape once and creates later plans of it by id."""
    d = _desc(c)
    if c["groups"] > 1:
        return b2c.Plan(d, b2c.POLICY_AUTO_TIMED, groups=c["groups"])
    key = bytes(d)
    if key not in _chosen:
        plan = b2c.Plan(d, b2c.POLICY_AUTO_TIMED)
        _chosen[key] = plan.info().id
        return plan
    return b2c.Plan(d, _chosen[key])


def _bytes(gen, shape, device="cuda"):
    return torch.randint(-128, 128, shape, dtype=torch.int8, device=device, generator=gen)


def _activations(gen, c, device="cuda"):
    shape = (c["C"], c["H"], c["W"]) if c["in_layout"] == b2c.LAYOUT_NCHW else (c["H"], c["W"], c["C"])
    return _bytes(gen, (c["N"],) + shape, device)


def _weights(gen, c):
    return _bytes(gen, (c["K"], c["C"] // c["groups"], c["R"], c["S"]))


def _outputs(c):
    P, Q = _out_extent(c)
    shape = (c["N"], c["K"], P, Q) if c["out_layout"] == b2c.LAYOUT_NCHW else (c["N"], P, Q, c["K"])
    y32 = torch.empty(shape, dtype=torch.int32, device="cuda") if c["out_mode"] & b2c.OUT_I32 else None
    y8 = torch.empty(shape, dtype=torch.int8, device="cuda") if c["out_mode"] & b2c.OUT_I8 else None
    return y32, y8


def _layer(gen, c):
    plan = _make_plan(c)
    plan.set_weights(_weights(gen, c))
    if c["act"]:
        reach = 1 << max(8, c["shift"] + 4)
        plan.set_activation(torch.randint(-reach, reach, (c["K"],), dtype=torch.int32, device="cuda", generator=gen), True)
    y32, y8 = _outputs(c)
    ws = torch.empty(max(16, plan.workspace_bytes()), dtype=torch.uint8, device="cuda")
    return {"plan": plan, "y32": y32, "y8": y8, "ws": ws}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    state = {"case": case}
    if case["kind"] == "stack":
        state["layers"] = [_layer(gen, c) for c in _layers(case)]
        state["x"] = _activations(gen, case)
    elif case["kind"] == "oneshot":
        state["x"], state["w"] = _activations(gen, case), _weights(gen, case)
        state["y32"], state["y8"] = _outputs(case)
        run(state)  # the first call of a shape selects its embedding
    elif case["kind"] == "stream":
        state.update(_layer(gen, case))
        host = torch.Generator()
        host.manual_seed(seed)
        P, Q = _out_extent(case)
        calls = range(case["calls"])
        # page-locked host buffers, as the streaming call asks for
        state["pinned"] = ([_activations(host, case, "cpu").pin_memory() for _ in calls],
                           [torch.empty((case["N"], case["K"], P, Q), dtype=torch.int8, pin_memory=True) for _ in calls])
        state["hx"] = [t.numpy() for t in state["pinned"][0]]
        state["hy"] = [t.numpy() for t in state["pinned"][1]]
    else:
        state.update(_layer(gen, case))
        state["x"] = _activations(gen, case)
    torch.cuda.synchronize()  # weights are in place before the first pass, whichever stream it uses
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "stack":
        x = state["x"]
        for layer in state["layers"]:
            layer["plan"].run(x, layer["y32"], layer["y8"], layer["ws"])
            x = layer["y8"]
        return [layer["y8"] if layer["y8"] is not None else layer["y32"] for layer in state["layers"]]
    if case["kind"] == "stream":
        for hx, hy in zip(state["hx"], state["hy"]):
            state["plan"].run_host_async(hx, None, hy)
        state["plan"].host_sync()
        return state["hy"]
    if case["kind"] == "oneshot":
        b2c.conv2d_int8(state["x"], state["w"], case["stride"], case["pad"], case["dil"], case["shift"], state["y32"],
                        state["y8"])
    else:
        state["plan"].run(state["x"], state["y32"], state["y8"], state["ws"])
    return [y for y in (state["y32"], state["y8"]) if y is not None]


def work(case):
    if case["kind"] == "stack":
        parts = [work(c) for c in _layers(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    P, Q = _out_extent(case)
    out = case["N"] * case["K"] * P * Q
    taps = case["C"] // case["groups"] * case["R"] * case["S"]
    per_out = (4 if case["out_mode"] & b2c.OUT_I32 else 0) + (1 if case["out_mode"] & b2c.OUT_I8 else 0)
    acts = case["N"] * case["C"] * case["H"] * case["W"] + out * per_out
    return {"bytes": case["calls"] * acts + case["K"] * taps, "flops": case["calls"] * 2 * out * taps}


def tolerance(case):
    # Sums of int8 products are exact in int32, and requantisation is integer arithmetic.
    return "exact"
