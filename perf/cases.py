"""Work that programs have this library do, for timing it and for comparing
its results: layers, blocks and whole networks run through the C ABI's Python
binding, with seeded inputs made on the GPU.

A case names a kind of work and its sizes; prepare() gives what a program
keeps between calls (weights loaded into an engine, device buffers), run() is
one call, exact() the same result in 64 bits from plain torch.
"""
import math

import torch

from paper_2401_16757_gb300 import capi

TORCH = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
SIZE = {"f32": 4, "f16": 2, "bf16": 2}


def listed():
    return [
        # the 6-layer fp32 perceptron at its batch of 8: the smallest call a
        # program makes, six short launches of a few MB of weights
        dict(name="mlp_f32_b8", kind="mlp", dtype="f32", rows=8, width=1024, depth=6),
        # the same network served at a larger, odd batch and a width that is
        # no multiple of a tile
        dict(name="mlp_f32_b100", kind="mlp", dtype="f32", rows=100, width=1000, depth=3),
        # the fully connected layers of VGG-16 at batch 16: a few rows
        # against 247 MB of weights
        dict(name="fc_f16_b16", kind="fc", dtype="f16", rows=16, feat=25088, hidden=4096, classes=1000),
        # a classifier layer through the allocation-free entry point
        dict(name="gemm_f16_b16", kind="gemm", dtype="f16", m=16, n=1000, k=2048, act=0),
        # a large projection through the same entry point
        dict(name="gemm_bf16_2048", kind="gemm", dtype="bf16", m=2048, n=4096, k=4096, act=1),
        # two bottlenecks of the last ResNet-50 stage on one image, the first
        # with its strided projection shortcut (latency)
        dict(name="bottlenecks_f16_b1", kind="bottlenecks", dtype="f16", batch=1, res=14, cin=1024, mid=512, stride=2),
        # two 3x3 convolutions and the pooling of a VGG-16 stage at batch 16
        dict(name="convs_f16_b16", kind="convs", dtype="f16", batch=16, res=56, cin=256, cout=256),
        # one layer of the 7B-shaped decoder over its 512-token prompt
        dict(name="prefill_bf16_512", kind="decoder", dtype="bf16", tokens=512, pos=0, max_seq=544, layers=1, d=4096,
             ffn=11008, vocab=0),
        # a ragged chunk of a prompt that continues a cached one, smaller model
        dict(name="prefill_bf16_79", kind="decoder", dtype="bf16", tokens=79, pos=100, max_seq=300, layers=2, d=1024,
             ffn=2752, vocab=0),
        # a whole greedy decode pass of a decoder at 7B width (two layers, the
        # embedding, the 32000-row head and the argmax) on a cache of 511
        dict(name="decode_bf16_d4096", kind="decoder", dtype="bf16", tokens=1, pos=511, max_seq=544, layers=2, d=4096,
             ffn=11008, vocab=32000),
        # block-swapped ResNet-50 on one image within 40 % of its weight bytes
        dict(name="resnet50_swapped", kind="resnet50", dtype="f16", batch=1, res=224, budget=0.4),
        # YOLOv3 on one image, all weights resident: 75 convolutions of every
        # size, upsampling, concatenation, three detection heads
        dict(name="yolov3_416", kind="yolov3", dtype="f16", batch=1, res=416, budget=0.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _candidate(rng):
    half = rng.choice(["f16", "bf16"])
    kind = rng.choice(["mlp", "mlp_batch", "fc", "gemm", "gemm_large", "bottlenecks", "convs", "prefill", "prefill",
                       "decode", "decode", "resnet50", "yolov3"])
    if kind == "mlp":
        return dict(kind="mlp", dtype="f32", rows=rng.randint(1, 16), width=4 * _log(rng, 64, 512), depth=rng.randint(2, 6))
    if kind == "mlp_batch":
        return dict(kind="mlp", dtype="f32", rows=_log(rng, 17, 512), width=_log(rng, 256, 2048), depth=rng.randint(1, 4))
    if kind == "fc":
        return dict(kind="fc", dtype=half, rows=_log(rng, 1, 64), feat=8 * _log(rng, 128, 3136),
                    hidden=8 * _log(rng, 64, 512), classes=rng.randint(10, 1000))
    if kind == "gemm":
        return dict(kind="gemm", dtype=half, m=_log(rng, 1, 64), n=_log(rng, 64, 4096), k=8 * _log(rng, 32, 512),
                    act=rng.randint(0, 2))
    if kind == "gemm_large":
        return dict(kind="gemm", dtype=half, m=_log(rng, 256, 4096), n=_log(rng, 512, 8192), k=8 * _log(rng, 64, 1024),
                    act=rng.randint(0, 2))
    if kind == "bottlenecks":
        mid = rng.choice([64, 128, 256, 512])
        return dict(kind="bottlenecks", dtype=half, batch=_log(rng, 1, 16), res=rng.randint(7, 56), cin=rng.choice([1, 2, 4]) * mid,
                    mid=mid, stride=rng.choice([1, 2]))
    if kind == "convs":
        c = rng.choice([64, 128, 256, 512])
        return dict(kind="convs", dtype=half, batch=_log(rng, 1, 16), res=2 * rng.randint(7, 56), cin=rng.choice([c // 2, c]),
                    cout=c)
    if kind in ("prefill", "decode"):
        tokens = 1 if kind == "decode" else _log(rng, 2, 512)
        d = rng.choice([512, 1024, 2048, 4096])
        pos = rng.randint(0, 1000)
        return dict(kind="decoder", dtype=half, tokens=tokens, pos=pos, max_seq=pos + tokens + rng.randint(0, 100),
                    layers=rng.randint(1, 2), d=d, ffn=8 * rng.randint(2 * d // 8, 11 * d // 32),
                    vocab=rng.choice([0, 8 * _log(rng, 128, 4000)]))
    if kind == "resnet50":
        return dict(kind=kind, dtype=half, batch=_log(rng, 1, 4), res=rng.randint(96, 224), budget=rng.choice([0.0, 0.4, 0.6]))
    return dict(kind=kind, dtype=half, batch=1, res=32 * rng.randint(7, 13), budget=rng.choice([0.0, 0.0, 0.3, 0.5]))


def draw(rng):
    most_flops = max(work(c)["flops"] for c in listed())
    most_bytes = max(work(c)["bytes"] for c in listed())
    while True:
        case = _candidate(rng)
        w = work(case)
        if w["flops"] <= most_flops and w["bytes"] <= most_bytes and _accepted(case):
            return case


def _accepted(case):
    """The allocation-free entry point refuses products whose partial sums exceed its 4 MiB of scratch."""
    if case["kind"] != "gemm":
        return True
    m, n, k = case["m"], case["n"], case["k"]
    splits = max(1, min(160 // (-(-m // 128) * -(-n // 64)), k // 128))
    return splits == 1 or splits * m * n * 4 <= 4 * 1024 * 1024 - 64 * 1024


# ------------------------------------------------------------ the networks
# A network is the binding's description of one: layers in execution order,
# each naming the layers that it reads (-1 is the input).
def _conv(src, cin, cout, k, stride=1, act="relu", res=None, res_post=False, gain=2.0):
    return dict(op="conv", src=[src], cin=cin, cout=cout, kh=k, kw=k, stride=stride, pad=k // 2, act=act, res=res,
                res_post=res_post, gain=gain)


def _linear(src, k, n, act="none", res=None, bias=True, gain=1.0):
    return dict(op="linear", src=[src], k=k, n=n, act=act, res=res, res_post=False, bias=bias, gain=gain)


def _bottleneck(layers, x, cin, mid, stride):
    layers.append(_conv(x, cin, mid, 1))
    layers.append(_conv(len(layers) - 1, mid, mid, 3, stride))
    main, short = len(layers) - 1, x
    if stride != 1 or cin != 4 * mid or x < 0:  # a shortcut is a layer's output
        layers.append(_conv(x, cin, 4 * mid, 1, stride, act="none"))
        short = len(layers) - 1
    # a small last gain in the residual branch keeps the sums of deep
    # networks in range, as a trained network's normalisation does
    layers.append(_conv(main, mid, 4 * mid, 1, res=short, gain=0.03))
    return len(layers) - 1


def _resnet50(case):
    layers = [_conv(-1, 3, 64, 7, 2), dict(op="maxpool", src=[0], kh=3, kw=3, stride=2, pad=1)]
    x, cin = 1, 64
    for blocks, mid, stride in ((3, 64, 1), (4, 128, 2), (6, 256, 2), (3, 512, 2)):
        for b in range(blocks):
            x = _bottleneck(layers, x, cin, mid, stride if b == 0 else 1)
            cin = 4 * mid
    layers.append(dict(op="gap", src=[x]))
    layers.append(_linear(len(layers) - 1, cin, 1000))
    return layers, [len(layers) - 1]


def _yolov3(case):
    layers, outs = [], []

    def conv(src, cin, cout, k, stride=1, act="leaky", res=None):
        layers.append(_conv(src, cin, cout, k, stride, act, res, True, gain=1.0))
        return len(layers) - 1

    x, c, route = conv(-1, 3, 32, 3), 32, {}
    for blocks, cout in ((1, 64), (2, 128), (8, 256), (8, 512), (4, 1024)):
        x, c = conv(x, c, cout, 3, 2), cout
        for _ in range(blocks):
            x = conv(conv(x, c, c // 2, 1), c // 2, c, 3, res=x)
        route[c] = x

    def head(x, cin, mid):
        x = conv(x, cin, mid, 1)
        x = conv(conv(x, mid, 2 * mid, 3), 2 * mid, mid, 1)
        branch = conv(conv(x, mid, 2 * mid, 3), 2 * mid, mid, 1)
        outs.append(conv(conv(branch, mid, 2 * mid, 3), 2 * mid, 255, 1, act="none"))
        return branch

    def up(branch, mid, other):
        u = conv(branch, mid, mid // 2, 1)
        layers.append(dict(op="upsample2x", src=[u]))
        layers.append(dict(op="concat", src=[len(layers) - 1, other]))
        return len(layers) - 1

    b = head(x, 1024, 512)
    b = head(up(b, 512, route[512]), 768, 256)
    head(up(b, 256, route[256]), 384, 128)
    return layers, outs


def _decoder(case):
    d, ffn, vocab = case["d"], case["ffn"], case["vocab"]
    layers, x = [], -1
    if vocab:
        layers.append(dict(op="embed", src=[-1], vocab=vocab, d=d))
        x = 0

    def add(layer):
        layers.append(layer)
        return len(layers) - 1

    def lin(src, k, n, act="none", res=None):
        return add(_linear(src, k, n, act, res, bias=False))

    for _ in range(case["layers"]):
        n = add(dict(op="rmsnorm", src=[x], d=d, eps=1e-6))
        q, k, v = lin(n, d, d), lin(n, d, d), lin(n, d, d)
        a = add(dict(op="attention", src=[q, k, v], heads=d // 128, max_seq=case["max_seq"], theta=10000.0))
        # the block input itself can only be a residual where it is a layer's output
        h = lin(a, d, d, res=x if x >= 0 else None)
        n = add(dict(op="rmsnorm", src=[h], d=d, eps=1e-6))
        g = lin(n, d, ffn)
        u = lin(n, d, ffn, "swiglu", g)
        x = lin(u, ffn, d, res=h)
    if not vocab:
        return layers, [x]
    n = add(dict(op="rmsnorm", src=[x], d=d, eps=1e-6))
    logits = lin(n, d, vocab)
    add(dict(op="argmax", src=[logits]))
    return layers, [logits, logits + 1]


def _model(case):
    kind = case["kind"]
    model = dict(name=kind, dtype=case["dtype"])
    if kind == "mlp":
        r, w, n = case["rows"], case["width"], case["depth"]
        model["input"] = (r, 1, 1, w)
        layers = [_linear(i - 1, w, w, "relu" if i < n - 1 else "none") for i in range(n)]
        outs = [n - 1]
    elif kind == "fc":
        model["input"] = (case["rows"], 1, 1, case["feat"])
        layers = [_linear(-1, case["feat"], case["hidden"], "relu", gain=2.0),
                  _linear(0, case["hidden"], case["hidden"], "relu", gain=2.0),
                  _linear(1, case["hidden"], case["classes"])]
        outs = [2]
    elif kind == "bottlenecks":
        model["input"] = (case["batch"], case["res"], case["res"], case["cin"])
        layers = []
        x = _bottleneck(layers, -1, case["cin"], case["mid"], case["stride"])
        outs = [_bottleneck(layers, x, 4 * case["mid"], case["mid"], 1)]
    elif kind == "convs":
        model["input"] = (case["batch"], case["res"], case["res"], case["cin"])
        layers = [_conv(-1, case["cin"], case["cout"], 3), _conv(0, case["cout"], case["cout"], 3),
                  dict(op="maxpool", src=[1], kh=2, kw=2, stride=2, pad=0)]
        outs = [2]
    elif kind == "decoder":
        layers, outs = _decoder(case)
        if case["vocab"]:
            model.update(input=(case["tokens"], 1, 1, 1), input_dtype="i32")
        else:
            model["input"] = (case["tokens"], 1, 1, case["d"])
    else:
        layers, outs = (_resnet50 if kind == "resnet50" else _yolov3)(case)
        model["input"] = (case["batch"], case["res"], case["res"], 3)
    model.update(layers=layers, outputs=outs)
    return model


def _shapes(model):
    """(n, h, w, c) of every layer's output."""
    got = []

    def of(i):
        return tuple(model["input"]) if i < 0 else got[i]

    for L in model["layers"]:
        n, h, w, c = of(L["src"][0])
        op = L["op"]
        if op in ("conv", "maxpool"):
            h = (h + 2 * L["pad"] - L["kh"]) // L["stride"] + 1
            w = (w + 2 * L["pad"] - L["kw"]) // L["stride"] + 1
            c = L.get("cout", c)
        elif op == "linear":
            h, w, c = 1, 1, L["n"]
        elif op == "gap":
            h = w = 1
        elif op == "upsample2x":
            h, w = 2 * h, 2 * w
        elif op == "concat":
            c += of(L["src"][1])[3]
        elif op == "embed":
            h, w, c = 1, 1, L["d"]
        elif op == "argmax":
            h, w, c = 1, 1, 1
        got.append((n, h, w, c))
    return got


def _tensors_of(L):
    """(shape, standard deviation) of a layer's parameter tensors, in storage order; a deviation of 0 means ones."""
    if L["op"] == "conv":
        fan = L["kh"] * L["kw"] * L["cin"]
        return [((L["cout"], L["kh"], L["kw"], L["cin"]), math.sqrt(L["gain"] / fan)), ((L["cout"],), 0.1)]
    if L["op"] == "linear":
        w = ((L["n"], L["k"]), 0.02 if not L["bias"] else math.sqrt(L["gain"] / L["k"]))
        return [w, ((L["n"],), 0.1)] if L["bias"] else [w]
    if L["op"] == "embed":
        return [((L["vocab"], L["d"]), 0.02 * 8)]
    if L["op"] == "rmsnorm":
        return [((L["d"],), 0.0)]
    return []


# ------------------------------------------------------------ inputs
def _rand(g, shape, std, dtype):
    t = torch.empty(shape, dtype=torch.float32, device="cuda")
    return t.normal_(0.0, std, generator=g).to(dtype)


def _inputs(case, seed):
    """The case's weights, input and cached keys and values, from the seed alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    dt = TORCH[case["dtype"]]
    if case["kind"] == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return dict(a=_rand(g, (m, k), 1.0, dt), w=_rand(g, (n, k), k ** -0.5, dt), bias=_rand(g, (n,), 0.1, dt))
    model = _model(case)
    got = dict(model=model, weights=[])
    for L in model["layers"]:
        got["weights"].append([_rand(g, shape, std, dt) if std else torch.ones(shape, dtype=dt, device="cuda")
                               for shape, std in _tensors_of(L)])
    if model["layers"][-1]["op"] == "argmax":
        # the head's rows differ in length, as a trained head's do: a few tokens stand out
        head = got["weights"][-2][0]
        head.copy_(head.float() * torch.exp(_rand(g, (head.shape[0], 1), 1.0, torch.float32)))
    if model.get("input_dtype") == "i32":
        got["x"] = torch.randint(0, case["vocab"], tuple(model["input"]), generator=g, device="cuda", dtype=torch.int32)
    else:
        got["x"] = _rand(g, tuple(model["input"]), 1.0, dt)
    if case["kind"] == "decoder":
        # per layer: keys (already rotated) and values of the cached positions
        cache = torch.zeros((case["layers"], 2, case["max_seq"], case["d"]), dtype=dt, device="cuda")
        cache[:, :, :case["pos"]] = _rand(g, (case["layers"], 2, case["pos"], case["d"]), 1.0, dt)
        got["cache"] = cache
    return got


def prepare(case, seed):
    inp = _inputs(case, seed)
    if case["kind"] == "gemm":
        inp["y"] = torch.empty((case["m"], case["n"]), dtype=TORCH[case["dtype"]], device="cuda")
        inp["args"] = (capi.DTYPE[case["dtype"]], inp["a"].data_ptr(), inp["w"].data_ptr(), inp["bias"].data_ptr(),
                       inp["y"].data_ptr(), case["m"], case["n"], case["k"], case["act"])
        return inp
    model, dt = inp["model"], TORCH[case["dtype"]]
    flat = [t for lw in inp["weights"] for t in lw]
    host = capi.HostWeights.allocate([t.numel() * t.element_size() for t in flat], pinned=True)
    for i, t in enumerate(flat):
        v = host.view(i)
        torch.from_numpy(v).copy_(t.reshape(-1).view(torch.uint8))
    desc = capi.Desc(model)
    if case.get("budget"):
        nbytes = sum(t.numel() * t.element_size() for t in flat)
        plan = capi.Plan.partition(desc, int(case["budget"] * nbytes), capi.options(swap_variant=capi.SWAP_ZEROCOPY))
    else:
        plan = capi.Plan.resident(desc)
    info = plan.info()
    st = dict(engine=capi.Engine(plan, host), plan=plan, x=inp["x"],
              out=torch.zeros(info["output_bytes"], dtype=torch.uint8, device="cuda"))
    shapes = _shapes(model)
    st["results"] = []
    for off, li in zip(plan.output_offsets(), model["outputs"]):
        n, h, w, c = shapes[li]
        whole = model["layers"][li]["op"] == "argmax"
        size = n * h * w * c * (4 if whole else SIZE[case["dtype"]])
        st["results"].append(st["out"][off:off + size].view(torch.int32 if whole else dt).view(n, h, w, c))
    if case["kind"] == "decoder":
        state = torch.zeros(info["state_bytes"], dtype=torch.uint8, device="cuda")
        st["position"] = state[:4].view(torch.int32)
        st["start"] = torch.tensor([case["pos"]], dtype=torch.int32, device="cuda")
        body = inp["cache"].reshape(-1).view(torch.uint8)  # rows of d * 2 bytes, d a multiple of 128: no gaps between caches
        assert info["state_bytes"] == 256 + body.numel()
        state[256:].copy_(body)
        st["state"] = state
        st["results"].append(state[256:].view(dt).view(inp["cache"].shape))
        st["engine"].bind_state(state.data_ptr(), info["state_bytes"])
    torch.cuda.synchronize()
    return st


def run(state):
    stream = torch.cuda.current_stream().cuda_stream
    if "args" in state:
        capi.gemm_noalloc(*state["args"], stream)
        return state["y"]
    if "position" in state:
        state["position"].copy_(state["start"])  # the sequence goes on from its cached prompt
    state["engine"].infer(state["x"].data_ptr(), state["out"].data_ptr(), stream)
    return state["results"]


# ------------------------------------------------------------ what a pass needs
def work(case):
    es = SIZE[case["dtype"]]
    if case["kind"] == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": es * (m * k + n * k + n + m * n), "flops": 2 * m * n * k}
    model = _model(case)
    shapes = _shapes(model)
    numel = [math.prod(s) for s in shapes]
    nbytes = math.prod(model["input"]) * (4 if "input_dtype" in model else es)
    flops = 0
    for i, L in enumerate(model["layers"]):
        if L["op"] == "embed":
            nbytes += case["tokens"] * L["d"] * es
            continue
        nbytes += es * sum(math.prod(shape) for shape, _ in _tensors_of(L))
        if L["op"] == "conv":
            flops += 2 * numel[i] * L["kh"] * L["kw"] * L["cin"]
        elif L["op"] == "linear":
            flops += 2 * numel[i] * L["k"]
        elif L["op"] == "attention":
            t, p, d = case["tokens"], case["pos"], case["d"]
            flops += 4 * d * (t * p + t * (t + 1) // 2)
            nbytes += 2 * es * d * (p + t)  # cached rows read, new rows written
    nbytes += sum(4 * numel[i] if model["layers"][i]["op"] == "argmax" else es * numel[i] for i in model["outputs"])
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the distance from the 64-bit result, which is what
    rounding every stored tensor to the storage type gives: 32-bit sums in
    any order for f32, one rounding per layer for the 16-bit types."""
    if case["dtype"] == "f32":
        return {"rel": 4e-6}
    deep = {"gemm": 1, "fc": 1.5, "convs": 1.5, "bottlenecks": 1.5, "decoder": 3, "resnet50": 3, "yolov3": 3.5}[case["kind"]]
    tol = {"rel": 1e-3 * deep if case["dtype"] == "f16" else 8e-3 * min(deep, 3)}
    if case["kind"] == "decoder" and case["vocab"]:
        tol["differ"] = 0.01  # greedy tokens where two logits are nearly equal
    return tol


# ------------------------------------------------------------ 64-bit results
def _act(v, act, res):
    if act == "relu":
        return v.clamp_min(0.0)
    if act == "leaky":
        return torch.where(v > 0, v, 0.1 * v)
    if act == "swiglu":
        return res * torch.sigmoid(res) * v
    return v


def _exact_conv(x, w, b, L):
    n, h, wd, c = x.shape
    p, s = L["pad"], L["stride"]
    oh, ow = (h + 2 * p - L["kh"]) // s + 1, (wd + 2 * p - L["kw"]) // s + 1
    xp = torch.nn.functional.pad(x, (0, 0, p, p, p, p))
    y = b.expand(n * oh * ow, -1).clone()
    for r in range(L["kh"]):
        for q in range(L["kw"]):
            t = xp[:, r:r + (oh - 1) * s + 1:s, q:q + (ow - 1) * s + 1:s, :]
            y.addmm_(t.reshape(-1, c), w[:, r, q, :].t())
    return y.view(n, oh, ow, -1)


def _rotate(v, pos, theta):
    """RoPE on adjacent pairs of every 128-wide head; v: [tokens, d]."""
    i = torch.arange(64, device="cuda", dtype=torch.float64)
    ang = pos[:, None].double() * theta ** (-2.0 * i / 128)
    cos, sin = ang.cos()[:, None, :], ang.sin()[:, None, :]
    p = v.view(v.shape[0], -1, 64, 2)
    a, b = p[..., 0], p[..., 1]
    return torch.stack((a * cos - b * sin, a * sin + b * cos), dim=-1).reshape(v.shape)


def _exact_attention(q, k, v, cache, case):
    t, p, d = case["tokens"], case["pos"], case["d"]
    pos = torch.arange(p, p + t, device="cuda")
    q, k = _rotate(q, pos, 10000.0), _rotate(k, pos, 10000.0)
    cache[0, p:p + t], cache[1, p:p + t] = k, v
    heads = d // 128
    keys = cache[0, :p + t].view(-1, heads, 128).permute(1, 0, 2)
    vals = cache[1, :p + t].view(-1, heads, 128).permute(1, 0, 2)
    s = q.view(t, heads, 128).permute(1, 0, 2) @ keys.transpose(1, 2) / math.sqrt(128.0)
    s = s.masked_fill(torch.arange(p + t, device="cuda")[None, :] > pos[:, None], -math.inf)
    return (torch.softmax(s, dim=-1) @ vals).permute(1, 0, 2).reshape(t, d)


def exact(case, seed):
    inp = _inputs(case, seed)
    if case["kind"] == "gemm":
        y = inp["bias"].double() + inp["a"].double() @ inp["w"].double().t()
        return _act(y, ("none", "relu", "leaky")[case["act"]], None)
    model = inp["model"]
    last = {}
    for i, L in enumerate(model["layers"]):
        for s in L["src"] + [L.get("res")]:
            last[s] = i
    cache = inp["cache"].double() if "cache" in inp else None
    got, attention = {-1: inp["x"] if "input_dtype" in model else inp["x"].double()}, 0
    for i, L in enumerate(model["layers"]):
        x, wb, op = got[L["src"][0]], [t.double() for t in inp["weights"][i]], L["op"]
        if op in ("conv", "linear"):
            res = None if L["res"] is None else got[L["res"]]
            if op == "conv":
                y = _exact_conv(x, wb[0], wb[1], L)
            else:
                y = x.reshape(x.shape[0], -1) @ wb[0].t()
                y = (y + wb[1] if len(wb) > 1 else y).view(x.shape[0], 1, 1, -1)
            if L["act"] == "swiglu":
                y = _act(y, "swiglu", res)
            elif res is not None and L["res_post"]:
                y = _act(y, L["act"], None) + res
            else:
                y = _act(y if res is None else y + res, L["act"], None)
        elif op == "maxpool":
            xc = torch.nn.functional.pad(x, (0, 0) + (L["pad"],) * 4, value=-math.inf)
            xc = xc.unfold(1, L["kh"], L["stride"]).unfold(2, L["kw"], L["stride"])
            y = xc.amax(dim=(-1, -2))
        elif op == "gap":
            y = x.mean(dim=(1, 2), keepdim=True)
        elif op == "upsample2x":
            y = x.repeat_interleave(2, dim=1).repeat_interleave(2, dim=2)
        elif op == "concat":
            y = torch.cat((x, got[L["src"][1]]), dim=3)
        elif op == "embed":
            y = wb[0][x.reshape(-1).long()].view(x.shape[0], 1, 1, -1)
        elif op == "rmsnorm":
            y = x / torch.sqrt(x.square().mean(dim=-1, keepdim=True) + L["eps"]) * wb[0]
        elif op == "attention":
            q, k, v = (got[s].view(case["tokens"], case["d"]) for s in L["src"])
            y = _exact_attention(q, k, v, cache[attention], case).view(case["tokens"], 1, 1, case["d"])
            attention += 1
        else:  # argmax: whole numbers, compared as they are
            y = None
        got[i] = y
        for s in list(got):
            if last.get(s, -1) <= i and s not in model["outputs"] and s != i:
                del got[s]
    outs = [got[i] for i in model["outputs"]]
    return outs + [cache] if cache is not None else outs
