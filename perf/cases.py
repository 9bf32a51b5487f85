"""The work that users of this library have it do, as cases that can be timed and compared.

Three kinds of program call it.  A serving loop runs packed layers: decode steps of one or a few rows, batches of
some tens to some hundreds of rows (continuous batching), prefill of hundreds to thousands of rows; through `Layer`
objects that it keeps, or, for the gated MLP, through `mlp_swiglu`; small decode steps often replayed from a CUDA
graph.  A conversion job quantises fp16 matrices and packs them.  An export job unpacks them again.

The layer shapes are those of `paper_2408_11743_b200/inputs.py`: K = N = 8192, the Llama-2-7B layers (hidden size
4096, intermediate size 11008) and the Llama-2-70B ones, and the column shards of the gate_up layer (22016 columns)
that tensor parallelism over four and eight GPUs leaves on each: 5504 and 2752 columns.  Values are drawn as there:
A ~ N(0, 1), codes uniform, scales uniform in [0.005, 0.02].
"""
import math

import torch

import paper_2408_11743_b200 as marlin

# the largest listed layer by weights and the largest listed pass by operations bound what draw() gives
MOST_WEIGHTS = 28672 * 8192
MOST_FLOPS = 2 * 2048 * 3 * 4096 * 11008


def listed():
    return [
        # one token through the smallest layer of a 7B model (o_proj), called from Python: latency of a call
        {"name": "decode-1-layer", "path": "layer", "format": "int4", "M": 1, "K": 4096, "N": 4096, "G": 128},
        # one token through the four layers of a 7B decoder block, replayed from a CUDA graph as serving loops do
        {"name": "decode-1-block", "path": "block", "M": 1, "K": 4096, "I": 11008, "G": 128, "graph": True},
        # sixteen sequences through the down projection of a 70B model with one scale per output channel
        {"name": "decode-16-channel", "path": "layer", "format": "int4", "M": 16, "K": 28672, "N": 8192, "G": 28672},
        # four sequences through an 8-bit layer
        {"name": "decode-4-w8", "path": "layer", "format": "w8", "M": 4, "K": 8192, "N": 8192, "G": 128},
        # thirty-two sequences through the layer of the batch sweep
        {"name": "batch-32-layer", "path": "layer", "format": "int4", "M": 32, "K": 8192, "N": 8192, "G": 128},
        # a continuous batch of an odd size through a 7B decoder block, called from Python
        {"name": "batch-100-block", "path": "block", "M": 100, "K": 4096, "I": 11008, "G": 128, "graph": False},
        # a batch through the 2:4 sparse layer
        {"name": "batch-64-sparse", "path": "layer", "format": "sparse24", "M": 64, "K": 8192, "N": 8192, "G": 128},
        # a batch through a layer with zero points, one of eight column shards of gate_up
        {"name": "batch-24-zp-shard", "path": "layer", "format": "zp", "M": 24, "K": 4096, "N": 2752, "G": 128},
        # prefill of a prompt of an odd length, one of four column shards of gate_up
        {"name": "prefill-777-shard", "path": "layer", "format": "int4", "M": 777, "K": 4096, "N": 5504, "G": 128},
        # prefill of a 2048-token prompt through the gated MLP of a 7B model
        {"name": "prefill-2048-mlp", "path": "mlp", "M": 2048, "K": 4096, "I": 11008, "G": 128},
        # conversion of the gate projection of a 7B model: quantise with the clipping search, then pack
        {"name": "convert-group", "path": "convert", "K": 4096, "N": 11008, "G": 128},
        # conversion of o_proj with one scale per output channel
        {"name": "convert-channel", "path": "convert", "K": 4096, "N": 4096, "G": 4096},
    ]


def _log_int(rng, low, high):
    return int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))


def _multiple(rng, low, high, of):
    return max(1, int(round(_log_int(rng, low, high) / of))) * of


def _columns(rng, low, high):
    # whole layers are multiples of 256 columns wide; shards of them need only be multiples of 64
    return _multiple(rng, low, high, 256 if rng.random() < 0.5 else 64)


def _group(rng, K, N):
    r = rng.random()
    if r < 0.6 or N % 256:
        return 128 if r < 0.8 else K
    return K if r < 0.8 else (64 if r < 0.9 else 32)


def draw(rng):
    path = rng.choices(["layer", "mlp", "block", "convert", "export"], [70, 8, 10, 8, 4])[0]
    while True:
        M = _log_int(rng, 1, 4096)
        if path == "mlp":
            case = {"path": path, "M": M, "K": _multiple(rng, 1024, 8192, 128), "I": _multiple(rng, 2048, 28672, 128), "G": 128}
        elif path == "block":
            M = min(_log_int(rng, 1, 256), 256)
            case = {"path": path, "M": M, "K": _multiple(rng, 1024, 8192, 128), "I": _multiple(rng, 2048, 28672, 128), "G": 128,
                    "graph": M <= 128 and rng.random() < 0.5}
        elif path in ("convert", "export"):
            K, N = _multiple(rng, 1024, 8192, 128), _columns(rng, 1024, 16384)
            case = {"path": path, "K": K, "N": N, "G": _group(rng, K, N)}
            if case["G"] == K > 4096:
                continue
        else:
            form = rng.choices(["int4", "zp", "w8", "sparse24"], [60, 15, 10, 15])[0]
            K = _multiple(rng, 1024, 28672, 128)
            N = _multiple(rng, 1024, 28672, 256) if form == "w8" else _columns(rng, 1024, 28672)
            case = {"path": path, "format": form, "M": M, "K": K, "N": N, "G": _group(rng, K, N)}
        if _weights(case) <= MOST_WEIGHTS and work(case)["flops"] <= MOST_FLOPS:
            return case


def _layers(case):
    """(K, N) of the products of a pass."""
    if case["path"] in ("layer", "convert", "export"):
        return [(case["K"], case["N"])]
    mlp = [(case["K"], 2 * case["I"]), (case["I"], case["K"])]
    return mlp if case["path"] == "mlp" else [(case["K"], 3 * case["K"]), (case["K"], case["K"])] + mlp


def _weights(case):
    return sum(K * N for K, N in _layers(case))


def work(case):
    """Bytes: weights, scales and what goes with them, activations and results, each once.  Operations: two per weight
    and row; of the quantiser about five per weight and candidate."""
    if case["path"] in ("convert", "export"):
        K, N, G = case["K"], case["N"], case["G"]
        codes, scales = K * N // 2, 2 * (K // G) * N
        if case["path"] == "export":
            return {"bytes": 2 * (codes + scales), "flops": 0}
        return {"bytes": 2 * K * N + 2 * (codes + scales), "flops": 5 * 10 * K * N}
    form, M, H, flops = case.get("format", "int4"), case["M"], case["K"], 0
    # columns of the activations read and of the results written; the intermediate of an MLP is neither
    nbytes = 2 * M * {"layer": H + case.get("N", 0), "mlp": 2 * H, "block": 7 * H}[case["path"]]
    for K, N in _layers(case):
        rows = 2 if form == "zp" else 1
        per = {"int4": K * N // 2, "zp": K * N // 2, "w8": K * N, "sparse24": K * N // 4 + K * N // 8}[form]
        nbytes += per + rows * 2 * (K // case["G"]) * N
        flops += 2 * M * K * N // (2 if form == "sparse24" else 1)
    return {"bytes": nbytes, "flops": flops}


class _Draws:
    """Seeded inputs on the GPU, of the distributions of `inputs.py`."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(seed)

    def normal(self, rows, cols, std=1.0):
        return torch.randn(rows, cols, generator=self.g, device="cuda").mul_(std).half()

    def codes(self, words, N):
        return torch.randint(-2 ** 31, 2 ** 31, (words, N), generator=self.g, device="cuda", dtype=torch.int32)

    def small(self, rows, N, below):
        return torch.randint(0, below, (rows, N), generator=self.g, device="cuda", dtype=torch.uint8)

    def scales(self, groups, N):
        return torch.rand(groups, N, generator=self.g, device="cuda").mul_(0.015).add_(0.005).half()

    def positions(self, K, N):
        keep = torch.tensor([(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)], device="cuda", dtype=torch.uint8)
        pattern = torch.randint(0, 6, (K // 4, N), generator=self.g, device="cuda")
        return keep[pattern].permute(0, 2, 1).reshape(K // 2, N).contiguous()


def _int4(d, K, N, G):
    return marlin.pack(d.codes(K // 8, N), d.scales(K // G, N), G)


def _layer(d, form, M, K, N, G):
    ws = marlin.new_workspace(M, K, N)
    if form == "int4":
        return marlin.Layer(*_int4(d, K, N, G), K, N, G, ws)
    if form == "zp":
        z = marlin.pack_zeros(d.small(K // G, N, 16), K, N, G)
        return marlin.Layer(*_int4(d, K, N, G), K, N, G, ws, z_packed=z)
    if form == "w8":
        return marlin.Layer(*marlin.pack_w8(d.small(K, N, 256), d.scales(K // G, N), G), K, N, G, ws, w8=True)
    w, meta, s = marlin.pack_sparse24(d.codes(K // 16, N), d.positions(K, N), d.scales(K // G, N), G)
    return marlin.Layer(w, s, K, N, G, ws, meta_packed=meta)


def prepare(case, seed):
    d, K, G = _Draws(seed), case["K"], case["G"]
    state = {"case": case}
    if case["path"] == "convert":
        state["W"] = d.normal(K, case["N"], 0.02)
        return state
    if case["path"] == "export":
        state["packed"] = _int4(d, K, case["N"], G)
        return state
    M = case["M"]
    state["x"] = d.normal(M, K)
    if case["path"] == "layer":
        state["layer"] = _layer(d, case["format"], M, K, case["N"], G)
        return state
    I = case["I"]
    # gate and up already interleaved: random codes are as good in any order; scales small enough for the intermediate
    gate_up = marlin.pack(d.codes(K // 8, 2 * I), d.scales(K // G, 2 * I).mul_(0.25), G)
    down = _int4(d, I, K, G)
    # one workspace of the largest size serves the layers of a model in turn
    sizes = [marlin.workspace_bytes(M, k, n) for k, n in _layers(case)]
    ws = torch.zeros(max(sizes), dtype=torch.uint8, device="cuda")
    state["mlp"] = (*gate_up, *down, K, I, K, G, ws)
    if case["path"] == "block":
        state["attended"], state["mlp_in"] = d.normal(M, K), d.normal(M, K)
        state["qkv"] = marlin.Layer(*_int4(d, K, 3 * K, G), K, 3 * K, G, ws)
        state["o_proj"] = marlin.Layer(*_int4(d, K, K, G), K, K, G, ws)
        if case["graph"]:
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                _block(state)
            torch.cuda.current_stream().wait_stream(side)
            state["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(state["graph"]):
                state["out"] = _block(state)
    return state


def _block(state):
    # the linear layers of one decoder block; what lies between them (attention, norms) is not this library's
    return {"qkv": state["qkv"](state["x"]), "o_proj": state["o_proj"](state["attended"]),
            "mlp": marlin.mlp_swiglu(state["mlp_in"], *state["mlp"])}


def run(state):
    case = state["case"]
    if case["path"] == "layer":
        return state["layer"](state["x"])
    if case["path"] == "mlp":
        return marlin.mlp_swiglu(state["x"], *state["mlp"])
    if case["path"] == "block":
        if case["graph"]:
            state["graph"].replay()
            return state["out"]
        return _block(state)
    if case["path"] == "convert":
        codes, scales = marlin.quantize_rtn(state["W"], case["G"])
        return (codes, scales, *marlin.pack(codes, scales, case["G"]))
    return marlin.unpack(*state["packed"], case["K"], case["N"], case["G"])


def tolerance(case):
    """Conversions are defined to the bit.  Products, measured against fp64 sums of the same weights over these ranges:
    relative 2-norm 2.1e-4 (the rounding of the fp16 results) to 2.9e-4 (where the scaled weights are rounded to fp16 as
    well), largest difference 1.2e-3; of the gated MLP, with its rounded intermediate, 5.1e-4 and 2.7e-3.  Four times
    that."""
    if case["path"] in ("convert", "export"):
        return "exact"
    if case["path"] == "layer":
        return {"rel": 1.15e-3, "max": 5e-3}
    return {"rel": 2e-3, "max": 1.1e-2}
