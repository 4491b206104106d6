"""Workloads for timing the library, through the calls a user's program makes.

Four kinds of work:
  net    a whole detector: pattern-pruned convolutions and the glue between them, one CUDA graph replayed per batch
         of frames (the network programs of this package)
  conv   one convolution call on the caller's tensors, issued call by call
  levels the independent convolutions of both detection towers on the five pyramid levels, one grouped call
  prune  one pruning iteration over a model that is being trained: select and pack every layer, then the masked
         dense weights W (.) M the next training step continues from, one CUDA graph per iteration

`listed()` holds the fixed cases, `draw()` gives more of the same ranges.  Inputs are made from a seed on the GPU:
activations ~N(0,1), Kaiming-normal weights, small biases.
"""
import math

import torch

from paper_2303_02191_b200 import binding as rt
from paper_2303_02191_b200 import retinanet_net, synth, yolov5s_net

TORCH_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
LAYOUT = {"nchw": rt.NCHW, "nhwc": rt.NHWC}
LEVELS = 5   # pyramid levels P3..P7


def listed():
    conv = dict(kind="conv", stride=1, bias=True, patterns="kernel")
    return [
        # a camera feeding single 640x640 frames: 57 small convolutions, latency and launch count decide
        dict(name="yolov5s_b1", kind="net", model="yolov5s", N=1, H=640, W=640, dtype="bf16", k=4),
        # the same detector on batches of frames (offline video, several cameras)
        dict(name="yolov5s_b16", kind="net", model="yolov5s", N=16, H=640, W=640, dtype="bf16", k=4),
        # the large detector at its usual frame size, batch 4: the largest case
        dict(name="retinanet_b4", kind="net", model="retinanet", N=4, H=800, W=1088, dtype="bf16", k=4),
        # the large detector on one small frame, fp16: maps down to 2x3 pixels, no layer fills the chip
        dict(name="retinanet_small", kind="net", model="retinanet", N=1, H=224, W=352, dtype="f16", k=3),
        # one fp32 layer on one small image in the default layout: the smallest call
        dict(conv, name="conv_f32_32ch", N=1, Cin=32, Cout=32, H=32, W=32, ksize=3, k=4, dtype="f32", layout="nchw", act="none"),
        # an ordinary detector layer, channels last
        dict(conv, name="conv_bf16_128ch", N=8, Cin=128, Cout=128, H=80, W=80, ksize=3, k=3, dtype="bf16", layout="nhwc", act="silu"),
        # the same layer for a program that keeps the default layout (NCHW)
        dict(conv, name="conv_bf16_128ch_nchw", N=8, Cin=128, Cout=128, H=80, W=80, ksize=3, k=2, dtype="bf16", layout="nchw", act="silu"),
        # full precision at a batch that fills the chip
        dict(conv, name="conv_f32_256ch_b32", N=32, Cin=256, Cout=256, H=80, W=80, ksize=3, k=4, dtype="f32", layout="nhwc", act="silu"),
        # channel counts and image sides that are multiples of nothing, as after channel pruning, fp16
        dict(conv, name="conv_f16_ragged", N=3, Cin=100, Cout=75, H=67, W=101, ksize=3, k=3, dtype="f16", layout="nhwc", act="relu"),
        # both detection towers on all pyramid levels at once, one pattern per block of filters x channels
        dict(name="towers_block_patterns", kind="levels", N=4, C=256, H=100, W=136, dtype="bf16", k=4, patterns="block"),
        # prune-retrain of the small detector: fp32 master weights, bf16 inference weights
        dict(name="prune_yolov5s", kind="prune", model="yolov5s", layers=0, Cin=0, Cout=0, k=4, w_dtype="f32", dtype="bf16"),
        # prune-retrain of the large detector: 32 M weights
        dict(name="prune_retinanet", kind="prune", model="retinanet", layers=0, Cin=0, Cout=0, k=4, w_dtype="f32", dtype="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["net", "net", "net", "conv", "conv", "conv", "conv", "levels", "prune", "prune"])
    if kind == "net":
        model = rng.choice(["yolov5s", "retinanet"])
        big = (16, 640, 640) if model == "yolov5s" else (4, 800, 1088)   # frame sides are multiples of 32
        return dict(kind="net", model=model, N=_log_int(rng, 1, big[0]), H=32 * rng.randint(3, big[1] // 32),
                    W=32 * rng.randint(3, big[2] // 32), dtype=rng.choice(["bf16", "bf16", "f16"]), k=rng.choice([2, 3, 4]))
    if kind == "conv":
        while True:
            c = dict(kind="conv", N=_log_int(rng, 1, 32), Cin=_log_int(rng, 3, 512), Cout=_log_int(rng, 16, 512),
                     H=_log_int(rng, 7, 160), W=_log_int(rng, 7, 160), ksize=rng.choice([3, 3, 1]), stride=rng.choice([1, 1, 2]),
                     k=rng.choice([2, 3, 4]), dtype=rng.choice(["bf16", "bf16", "f16", "f32"]),
                     layout=rng.choice(["nhwc", "nhwc", "nchw"]), act=rng.choice(["silu", "relu", "none"]),
                     bias=rng.random() < 0.8, patterns="kernel")
            if rng.random() < 0.7:      # most layers have channel counts that are multiples of 16
                c["Cin"], c["Cout"] = max(16, c["Cin"] // 16 * 16), max(16, c["Cout"] // 16 * 16)
            if c["ksize"] == 3 and c["Cin"] % 16 == 0 and rng.random() < 0.2:
                c["patterns"] = "block"
            w = work(c)
            if w["flops"] <= 110e9 and w["bytes"] <= 1.5e9:
                return c
    if kind == "levels":
        return dict(kind="levels", N=_log_int(rng, 1, 4), C=16 * rng.randint(4, 16), H=rng.randint(13, 100), W=rng.randint(13, 136),
                    dtype=rng.choice(["bf16", "f16"]), k=rng.choice([2, 3, 4]), patterns=rng.choice(["kernel", "block"]))
    c = dict(kind="prune", model=rng.choice(["yolov5s", "retinanet", "plain", "plain"]), layers=0, Cin=0, Cout=0,
             k=rng.choice([2, 3, 4, 5]), w_dtype=rng.choice(["f32", "f32", "bf16", "f16"]), dtype=rng.choice(["bf16", "bf16", "f16", "f32"]))
    if c["model"] == "plain":   # a stack of alternating 3x3 and 1x1 layers of one width
        c.update(layers=_log_int(rng, 2, 50), Cin=_log_int(rng, 16, 400), Cout=_log_int(rng, 16, 400))
    return c


# ---- inputs ---------------------------------------------------------------------------------------------------

_CTX = []


def _ctx():
    """The one context a program keeps per device."""
    if not _CTX:
        _CTX.append(rt.Context(0))
    return _CTX[0]


def _masks(k):
    return rt.rtoss_pattern_preset(k, {4: rt.PRESET_CENTRE8, 9: rt.PRESET_DENSE}.get(k, rt.PRESET_CONN4))


class _Rand:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed))

    def normal(self, shape, std, dtype=torch.float32):
        return torch.empty(shape, dtype=torch.float32, device="cuda").normal_(0.0, std, generator=self.g).to(dtype)

    def weights(self, cout, cin, ksize, dtype=torch.float32):
        return self.normal((cout, cin, ksize, ksize), math.sqrt(2.0 / (cin * ksize * ksize)), dtype)


def _packed(rand, cout, cin, ksize, k, dtype, patterns="kernel"):
    ctx, masks, w = _ctx(), _masks(k), rand.weights(cout, cin, ksize)
    if patterns == "block":
        pid = ctx.rtoss_select_patterns_shared(w, masks, k, 128, 16)
    else:
        pid = ctx.rtoss_select_patterns(w, ksize, masks, k)
    return ctx.rtoss_pack(w, ksize, masks, k, pid, rt.DTYPE_NAMES[dtype])


def _shape(layout, N, C, H, W):
    return (N, H, W, C) if layout == "nhwc" else (N, C, H, W)


def _level_sizes(case):
    H, W, got = case["H"], case["W"], []
    for _ in range(LEVELS):
        got.append((H, W))
        H, W = synth.out_hw(H, W, 2)
    return got


def _prune_layers(case):
    if case["model"] == "yolov5s":
        return [(L["cout"], L["cin"], L["ksize"]) for L in synth.yolov5s_stack()]
    if case["model"] == "retinanet":
        return list({L["wid"]: (L["cout"], L["cin"], L["ksize"]) for L in synth.retinanet_r50fpn_stack()}.values())
    return [(case["Cout"], case["Cin"], 3 if i % 2 == 0 else 1) for i in range(case["layers"])]


def _graph(fn):
    """fn captured once, as a program that repeats it would keep it."""
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        fn()
    torch.cuda.current_stream().wait_stream(side)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fn()
    return g


def prepare(case, seed):
    ctx, rand, kind = _ctx(), _Rand(seed), case["kind"]
    if kind == "net":
        mod = yolov5s_net if case["model"] == "yolov5s" else retinanet_net
        net = mod.GpuNet(ctx, case["N"], case["H"], case["W"], k=case["k"], seed=int(seed) % (1 << 31), dtype=case["dtype"])
        x = net.t["in"]
        x.copy_(rand.normal(x.shape, 1.0, x.dtype))
        net.run()   # finds out which fused calls the library takes
        graph = _graph(lambda: net.run(chained=True))
        names = yolov5s_net.OUTPUTS if case["model"] == "yolov5s" else net.output_names
        return dict(kind=kind, net=net, graph=graph, out=[net.t[n] for n in names])
    if kind == "conv":
        td = TORCH_DTYPE[case["dtype"]]
        Ho, Wo = synth.out_hw(case["H"], case["W"], case["stride"])
        return dict(kind=kind, call=ctx.rtoss_conv3x3_pattern if case["ksize"] == 3 else ctx.rtoss_conv1x1_pattern,
                    packed=_packed(rand, case["Cout"], case["Cin"], case["ksize"], case["k"], case["dtype"], case["patterns"]),
                    x=rand.normal(_shape(case["layout"], case["N"], case["Cin"], case["H"], case["W"]), 1.0, td),
                    y=torch.empty(_shape(case["layout"], case["N"], case["Cout"], Ho, Wo), dtype=td, device="cuda"),
                    bias=rand.normal((case["Cout"],), 0.1) if case["bias"] else None,
                    args=(case["N"], case["H"], case["W"], case["stride"], LAYOUT[case["layout"]], rt.ACT_NAMES[case["act"]]))
    if kind == "levels":
        td, C, N = TORCH_DTYPE[case["dtype"]], case["C"], case["N"]
        keep, items, out = [], [], []
        feats = [rand.normal((N, h, w, C), 1.0, td) for h, w in _level_sizes(case)]   # both towers read the same level
        for _ in range(2):
            packed, bias = _packed(rand, C, C, 3, case["k"], case["dtype"], case["patterns"]), rand.normal((C,), 0.1)
            keep += [packed, bias]
            for x in feats:
                y = torch.empty_like(x)
                items.append(ctx.conv_item(packed, x, y, N, x.shape[1], x.shape[2], 1, rt.NHWC, rt.ACT_RELU, bias))
                out.append(y)
        return dict(kind=kind, items=items, out=out, keep=keep + feats)
    # prune
    masks, td = _masks(case["k"]), TORCH_DTYPE[case["dtype"]]
    items, handles, at_pid, at_w = [], [], 0, 0
    for cout, cin, ks in _prune_layers(case):
        n_w = cout * cin * ks * ks
        items.append(dict(w=rand.weights(cout, cin, ks, TORCH_DTYPE[case["w_dtype"]]), ksize=ks, masks=masks, k=case["k"],
                          at=(at_pid, n_w // 9, at_w)))
        at_pid += (n_w // 9 + 255) // 256 * 256
        at_w += (n_w + 127) // 128 * 128
    pids = torch.zeros(max(at_pid, 1), dtype=torch.uint8, device="cuda")
    dense = torch.zeros(at_w, dtype=td, device="cuda")
    for it in items:
        a, n, b = it.pop("at")
        it["pid"] = pids[a:a + n]
        pid = ctx.rtoss_select_patterns(it["w"], it["ksize"], masks, case["k"], pid=it["pid"])
        it["packed"] = ctx.rtoss_pack(it["w"], it["ksize"], masks, case["k"], pid, rt.DTYPE_NAMES[case["dtype"]])
        handles.append((it["packed"], dense[b:]))
    batch = ctx.rtoss_batch_create(items)

    def iteration():
        batch.rtoss_batch_select_pack()
        stream = torch.cuda.current_stream().cuda_stream
        for packed, out in handles:
            ctx._check(rt.lib.rtoss_packed_to_dense(ctx.h, packed.h, out.data_ptr(), stream))

    return dict(kind=kind, batch=batch, graph=_graph(iteration), keep=(items, handles), out=[pids, dense])


def run(state):
    kind = state["kind"]
    if kind == "conv":
        return state["call"](state["packed"], state["x"], state["y"], *state["args"], bias=state["bias"])
    if kind == "levels":
        _ctx().rtoss_conv_group(state["items"])
    else:
        state["graph"].replay()
    return state["out"]


# ---- what a pass cannot do without, and how exact it has to be ---------------------------------------------------

def work(case):
    """Inputs once, weights once in packed form, outputs once; operations on the kept weights only.  What a network
    passes from layer to layer is not counted as bytes."""
    kind, k = case["kind"], case["k"]
    if kind == "prune":
        n = sum(cout * cin * ks * ks // 9 for cout, cin, ks in _prune_layers(case))
        we, e, P = (4 if case["w_dtype"] == "f32" else 2), (4 if case["dtype"] == "f32" else 2), len(_masks(k))
        return dict(bytes=n * (9 * we + 1 + k * e + 9 * e), flops=n * (9 + P * (k - 1)))
    e, N = 4 if case["dtype"] == "f32" else 2, case["N"]
    if kind == "net":
        layers = (synth.yolov5s_stack if case["model"] == "yolov5s" else synth.retinanet_r50fpn_stack)(case["H"], case["W"])
        flops = sum(synth.layer_nnz_flops(L, N, k) for L in layers)
        wts = {L["wid"]: L["cout"] * L["cin"] * L["ksize"] ** 2 // 9 * (k * e + 1) + 4 * L["cout"] for L in layers}
        if case["model"] == "yolov5s":
            n_in = 3 * case["H"] * case["W"]
            n_out = sum(c * (case["H"] // s) * (case["W"] // s) for c, s in ((128, 8), (256, 16), (512, 32)))
        else:
            n_in = 64 * (case["H"] // 4) * (case["W"] // 4)
            n_out = sum(256 * L["H"] * L["W"] for L in layers if "_tower3." in L["name"])
        return dict(bytes=N * (n_in + n_out) * e + sum(wts.values()), flops=flops)
    if kind == "levels":
        layers = [dict(cin=case["C"], cout=case["C"], ksize=3, stride=1, H=h, W=w) for h, w in _level_sizes(case)]
        w1 = case["C"] ** 2 * (k * e + 1) + 4 * case["C"]
        pix = sum(h * w for h, w in _level_sizes(case))
        return dict(bytes=3 * N * pix * case["C"] * e + 2 * w1, flops=2 * sum(synth.layer_nnz_flops(L, N, k) for L in layers))
    L = dict(cin=case["Cin"], cout=case["Cout"], ksize=case["ksize"], stride=case["stride"], H=case["H"], W=case["W"])
    return dict(bytes=synth.layer_bytes(L, N, k, e), flops=synth.layer_nnz_flops(L, N, k))


def tolerance(case):
    """About four times what a pass differs by from the same pass summed in 64 bits (networks: with every layer's
    result rounded to the data type, as the library rounds it)."""
    kind, dt = case["kind"], case["dtype"]
    if kind == "prune":
        return "exact"
    if kind == "net":       # a one-ulp flip in a layer spreads through the layers behind it
        if case["model"] == "yolov5s":
            return {"rel": 0.01, "max": 0.06} if dt == "bf16" else {"rel": 0.0014, "max": 0.007}
        return {"rel": 0.02, "max": 0.25} if dt == "bf16" else {"rel": 0.006, "max": 0.045}
    if dt == "f32":         # FMA sums in the default layout; split tf32 products where channels come last
        return {"rel": 1e-5, "max": 4e-5} if case["layout"] == "nchw" else {"rel": 8e-5, "max": 3e-4}
    if dt == "bf16":
        return {"rel": 5e-4, "max": 0.03}
    silu = case.get("act") == "silu"   # its approximation is as coarse as an fp16 result's last bit
    return {"rel": 3e-4 if silu else 1e-4, "max": 0.004}
