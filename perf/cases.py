"""Performance cases of the library: the work that a program built on it has it do.

Most cases are decode steps: every linear layer of one or more decoder layers, called through the public entry
points with buffers that such a program allocates once. Layer shapes are those of the benchmark configurations
(written N x K, rows x input channels); the ragged case and the drawn ones are generic. As many decoder layers as
it takes go into one pass for the weights to exceed the L2 cache, as they do in a real step. The other cases are
what surrounds decoding: quantizing the activations of a whole prompt, and the export of a trained layer to packed
codes and grids.
"""
import math

import torch

import paper_2502_15779_b200 as rcp

DEV = "cuda:0"

# (rows x input channels) of the linear layers of one decoder layer
L_1B = "2048x2048,512x2048,512x2048,2048x2048,8192x2048,8192x2048,2048x8192"
L_7B = "12288x4096,4096x4096,22016x4096,4096x11008"
L_8B = "6144x4096,4096x4096,28672x4096,4096x14336"
L_70B = "10240x8192,8192x8192,57344x8192,8192x28672"


def _case(name, op, M, shapes, layers, group=0, graph=False):
    return {"name": name, "op": op, "M": M, "shapes": shapes, "layers": layers, "group": group, "graph": graph}


def listed():
    return [
        # one small projection on its own, one token: nothing but latency
        _case("single_2048_m1", "linear", 1, "2048x2048", 1),
        # a whole decode step of a small model (sixteen layers, one token), captured once and replayed, as a program
        # does where launches would bound it; the other steps marked `graph` likewise
        _case("decode_1b_m1_graph", "linear", 1, L_1B, 16, graph=True),
        # one token through the layers of the common model sizes: the setting of the paper's own kernel
        _case("decode_7b_m1_graph", "linear", 1, L_7B, 4, graph=True),
        _case("decode_70b_m1", "linear", 1, L_70B, 1),
        # rows and channels that divide nothing, a few tokens in flight
        _case("ragged_m3", "linear", 3, "5003x2624,1777x11008,10007x4096,333x5184,4100x8192", 4),
        # batched decoding: a full batch on a mid-sized model, eight sequences on the largest
        _case("decode_8b_m16", "linear", 16, L_8B, 2),
        _case("decode_70b_m8", "linear", 8, L_70B, 1),
        # the paper's own granularity, one grid per 128 weights
        _case("grouped_8b_m1_graph", "linear", 1, L_8B, 4, group=128, graph=True),
        # weight-only setting: activations stay in 16 bits
        _case("w2a16_8b_m2", "w2a16", 2, L_8B, 4),
        # 3-bit setting, one token
        _case("w3a4_8b_m1", "w3a4", 1, L_8B, 2),
        # activations of a prompt of 2048 tokens, rotated and quantized: attention and MLP inputs, down projection
        _case("prefill_quantize_8b", "quantize", 2048, "0x4096,0x4096,0x14336", 1),
        # offline: a trained layer turned into packed codes and group-wise grids
        _case("export_8b_layer", "ldp_export", 0, L_8B, 1, group=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: sizes spread over their logarithm, odd row counts among them."""
    op = rng.choice(["linear"] * 6 + ["w2a16", "w3a4", "quantize", "ldp_export"])
    group = 0
    if op == "linear":
        group = rng.choice([0, 0, 128])
        M = rng.choice([1, 1, rng.randint(2, 16)])
    elif op == "w2a16":
        M = rng.randint(1, 4)
    elif op == "w3a4":
        M, group = rng.choice([1, 1, 2]), rng.choice([0, 128])
    elif op == "quantize":
        M = _log_int(rng, 1, 4096)
    else:
        M, group = 0, 128
    shapes, total = [], 0
    # no drawn case is larger than the largest listed one of its kind
    cap = 1 << 27 if op == "ldp_export" else min(856 << 20, int(6.7e9) // max(M, 1))
    for _ in range(rng.randint(1, 4)):
        if rng.random() < 0.5:
            K = rng.choice([2048, 4096, 8192, 11008, 14336, 28672])
        else:
            K = 128 * _log_int(rng, 4, 112)
        N = 0
        if op != "quantize":
            N = _log_int(rng, 256, 57344 * 8192 // max(K, 8192))
            N = max(1, min(N, (cap - total) // K))
            if rng.random() < 0.5:
                N = max(128, N // 128 * 128)
        if total and total + N * K > cap:
            break
        total += N * K
        shapes.append("%dx%d" % (N, K))
    # a few decoder layers, so that the weights come from memory as they do in a step
    layers = 1 if op in ("quantize", "ldp_export") else max(1, min(8, cap // total, (1 << 29) // total))
    c = _case("", op, M, ",".join(shapes), layers, group, op == "linear" and rng.random() < 0.3)
    del c["name"]
    return c


def _shapes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split(",")]


def _had_block(K):
    """Rotation block: the whole token where its length is a power of two, 128 (or what divides it) otherwise."""
    if K & (K - 1) == 0 and K <= 8192:
        return K
    return 128 if K % 128 == 0 else 64


def _codes(N, K, three, g):
    """Codes of a trained layer: the inner levels are met more often than the outer ones."""
    out = torch.randint(0, 256, (N, K), generator=g, device=DEV, dtype=torch.uint8)
    steps = (38, 127, 217) if not three else (12, 44, 84, 127, 171, 211, 243)
    codes = torch.zeros_like(out)
    for t in steps:
        codes += out > t
    return codes


def _levels(shape, n, g):
    lv = torch.randn(*shape, n, generator=g, device=DEV) * 0.02
    return torch.sort(lv, dim=-1)[0].to(torch.float16).contiguous()


def _activations(M, K, g):
    """Normal with one element in a hundred twenty times as large: what rotation is there for."""
    x = torch.randn(M, K, generator=g, device=DEV)
    hit = torch.rand(M, K, generator=g, device=DEV) < 0.01
    return torch.where(hit, x * 20.0, x).to(torch.float16).contiguous()


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    op, M, group = case["op"], case["M"], case["group"]
    items = []
    # results of a linear layer, one buffer for all decoder layers of the step
    ys = [torch.empty(case["layers"], max(M, 1), N, dtype=torch.float16, device=DEV) for N, K in _shapes(case)]
    for layer in range(case["layers"]):
        for (N, K), y in zip(_shapes(case), ys):
            it = {"B": _had_block(K)}
            if op == "ldp_export":
                it["w"] = (torch.randn(N, K, generator=g, device=DEV) * 0.02).to(torch.float16)
                it["sig"] = [torch.sigmoid(torch.randn(N, K // group, generator=g, device=DEV) * 0.3 + b).contiguous()
                             for b in (3.0, 3.0, -0.7, 0.0)]
                items.append(it)
                continue
            it["x"] = _activations(M, K, g)
            if op in ("linear", "w3a4", "quantize"):
                it["xq"] = torch.empty(M, K // 2, dtype=torch.uint8, device=DEV)
                it["scale"] = torch.empty(M, dtype=torch.float16, device=DEV)
            if op != "quantize":
                three = op == "w3a4"
                codes = _codes(N, K, three, g)
                if three:
                    it["words2"], it["words1"] = rcp.rcp_pack_weights3(codes)
                else:
                    it["words"] = rcp.rcp_pack_weights(codes)
                del codes
                it["lut"] = _levels((N,) if group == 0 else (N, K // group), 8 if three else 4, g)
                it["y"] = y[layer]
                if not three:
                    it["ws"] = rcp.make_workspace(M, N, K, DEV)
                if op == "w2a16":
                    it["digits"] = torch.empty(M, 4, K, dtype=torch.int8, device=DEV)
                    it["unit"] = torch.empty(M, 4, dtype=torch.float32, device=DEV)
            items.append(it)
    state = {"case": case, "items": items, "ys": ys, "graph": None}
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _step(state)
        torch.cuda.current_stream().wait_stream(side)
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            _step(state)
    return state


def _step(state):
    op, group = state["case"]["op"], state["case"]["group"]
    if op == "quantize":
        return [rcp.rcp_quantize_act(it["x"], it["B"], 1.0, xq=it["xq"], scale=it["scale"]) for it in state["items"]]
    if op == "ldp_export":
        return [rcp.rcp_ldp_export(it["w"], *it["sig"], group) for it in state["items"]]
    for it in state["items"]:
        if op == "linear":
            rcp.rcp_linear_w2a4(it["x"], it["B"], 1.0, it["words"], it["lut"], group=group, y=it["y"], xq=it["xq"],
                                scale=it["scale"], workspace=it["ws"])
        elif op == "w2a16":
            rcp.rcp_gemv_w2a16(it["words"], it["lut"], it["x"], y=it["y"], digits=it["digits"], unit=it["unit"],
                               workspace=it["ws"])
        else:
            rcp.rcp_quantize_act(it["x"], it["B"], 1.0, xq=it["xq"], scale=it["scale"])
            rcp.rcp_gemv_w3a4(it["words2"], it["words1"], it["lut"], it["xq"], it["scale"], group=group, y=it["y"])
    return state["ys"]


def run(state):
    if state["graph"] is None:
        return _step(state)
    state["graph"].replay()
    return state["ys"]


def work(case):
    op, M, group = case["op"], case["M"], case["group"]
    nbytes = flops = 0
    for N, K in _shapes(case):
        if op == "quantize":
            nbytes += 2 * M * K + M * K // 2 + 2 * M
            flops += M * K * (int(math.log2(_had_block(K))) + 3)
        elif op == "ldp_export":
            units = N * (K // group)
            nbytes += 2 * N * K + 16 * units + N * K // 4 + 8 * units
            flops += 6 * N * K
        else:
            three = op == "w3a4"
            units = N if group == 0 else N * (K // group)
            nbytes += (3 * N * K // 8 + 16 * units if three else N * K // 4 + 8 * units) + 2 * M * K + 2 * M * N
            flops += 2 * M * N * K
    return {"bytes": nbytes * case["layers"], "flops": flops * case["layers"]}


def tolerance(case):
    if case["op"] in ("quantize", "ldp_export"):
        return "exact"
    # whole-number sums, a few fp32 operations, one rounding to fp16: four times what that rounding alone gives
    # (against the same in 64 bits: 2.1e-4 in the 2-norm, 4.9e-4 at most)
    return {"rel": 8e-4, "max": 2e-3}
