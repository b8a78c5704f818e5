"""The work that users of this package have it do, as cases that can be timed.

Kinds of case:
  call      one eager call of ptqtp_gemv on one matrix (a program that does not capture its decode step)
  host      one ptqtp_gemv_host call: activations in pinned host memory, the result read on the host
  layer     one decode step over a few decoder layers, captured once as a CUDA graph and replayed, as a decoder does:
            per layer the q, k, v, o, gate, up and down projections at batch m
              form "separate": seven ptqtp_gemv calls, every projection with activations of its own
              form "fused":    ptqtp_gemv_multi (q, k, v), ptqtp_gemv (o), ptqtp_gemv_multi (gate, up, gated pair),
                               ptqtp_gemv (down), each on the result of the one before
              form "skinny":   seven ptqtp_gemm_skinny calls (m >= 2)
              form "ws":       seven ptqtp_gemm_skinny_ws calls with one workspace (format 2, m >= 2)
  pack      ptqtp_pack of one matrix; unpack: its inverse
  quantise  ptqtp_decompose of a weight matrix and ptqtp_pack of the planes, as a conversion program does per matrix

The shapes are those of inputs.py (LLaMA-3-8B, LLaMA-3-70B, Qwen3-0.6B) or generic; planes, scales and activations
follow the distributions of inputs.py, drawn on the device.
"""
import torch

from paper_2509_16989_b200 import binding
from paper_2509_16989_b200.inputs import LLAMA3_8B, LLAMA3_70B, QWEN3_0P6B_UP, make_weights_device

GROUP = 128


def _dims(shapes):
    return {"hidden": shapes["q"][1] if "q" in shapes else shapes["qo"][1],
            "kv": shapes["k"][0] if "k" in shapes else shapes["kv"][0],
            "inter": shapes["gate"][0] if "gate" in shapes else shapes["gate_up"][0]}


def _layer(name, shapes, layers, m, form, fmt, level, p_zero=0.4):
    return {"name": name, "kind": "layer", **_dims(shapes), "layers": layers, "m": m, "form": form, "fmt": fmt,
            "level": level, "p_zero": p_zero}


def listed():
    n_up, k_up = QWEN3_0P6B_UP
    return [
        # the smallest calls: one matrix of a small model at the library's default settings
        {"name": "call_small", "kind": "call", "n": n_up, "k": k_up, "fmt": 3},
        # a matrix that no tile size divides, on the binding's default format
        {"name": "call_ragged", "kind": "call", "n": 5003, "k": 6272, "fmt": 2},
        # a caller whose activations live on the host
        {"name": "host_4096", "kind": "host", "n": LLAMA3_8B["q"][0], "k": LLAMA3_8B["q"][1], "fmt": 3},
        # single-sequence decode, one call per matrix: the benchmark's headline step
        _layer("decode_8b", LLAMA3_8B, 2, 1, "separate", 3, 2),
        # single-sequence decode in four launches per layer, each waiting for the result of the one before
        _layer("decode_8b_fused", LLAMA3_8B, 2, 1, "fused", 3, 1),
        # serving a few sequences together on the blobs of the decoder
        _layer("batch4_8b", LLAMA3_8B, 2, 4, "skinny", 3, 2),
        _layer("batch16_8b", LLAMA3_8B, 2, 16, "skinny", 3, 0),
        # the largest batch that the library takes
        _layer("batch64_8b", LLAMA3_8B, 2, 64, "skinny", 3, 0),
        # a large model at batch 8 with the workspace call on the default format
        _layer("batch8_70b", LLAMA3_70B, 1, 8, "ws", 2, 0, p_zero=0.5),
        # conversion of a checkpoint and back
        {"name": "pack_gate", "kind": "pack", "n": LLAMA3_8B["gate"][0], "k": LLAMA3_8B["gate"][1], "fmt": 3},
        {"name": "unpack_down", "kind": "unpack", "n": LLAMA3_8B["down"][0], "k": LLAMA3_8B["down"][1], "fmt": 2},
        {"name": "quantise_gate", "kind": "quantise", "n": LLAMA3_8B["gate"][0], "k": LLAMA3_8B["gate"][1], "fmt": 3},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _cols(rng, lo, hi):
    """A number of columns: a multiple of the scale group, and of nothing more."""
    return max(1, round(_log(rng, lo, hi) / GROUP)) * GROUP


def draw(rng):
    kind = rng.choice(["call", "host", "layer", "layer", "layer", "layer", "pack", "unpack", "quantise"])
    if kind == "layer":
        hidden = _cols(rng, 1024, 6144)
        case = {"kind": kind, "hidden": hidden, "kv": hidden // rng.choice([1, 2, 4, 8]) if hidden < 4096 else hidden // 8,
                "inter": round(hidden * rng.uniform(2.5, 4.0) / GROUP) * GROUP,
                "layers": rng.choice([1, 2]) if hidden < 4096 else 1, "p_zero": rng.choice([0.4, 0.5])}
        form = rng.choice(["separate", "fused", "skinny", "skinny", "skinny", "ws"])
        if form == "separate":
            return {**case, "m": 1, "form": form, "fmt": rng.choice([2, 3, 3]), "level": rng.choice([0, 2, 2])}
        if form == "fused":
            return {**case, "m": 1, "form": form, "fmt": 3, "level": rng.choice([0, 1])}
        # several rows on format 2 take a pass per four rows without a workspace: its callers keep to a few rows
        fmt = 2 if form == "ws" else rng.choice([2, 3, 3, 3])
        most = 4 if form == "skinny" and fmt == 2 else 64 if hidden < 4096 else 48
        return {**case, "m": _log(rng, 2, most), "form": form, "fmt": fmt, "level": rng.choice([0, 2])}
    n, k = _log(rng, 1024, 14336), _cols(rng, 1024, 4096 if kind == "quantise" else 14336)
    return {"kind": kind, "n": n, "k": k, "fmt": rng.choice([2, 3])}


# ---- inputs ----

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _trits(g, n, k, p_zero):
    # P(-1) = P(+1) = (1 - p_zero) / 2, in thousandths
    r = torch.randint(0, 1000, (n, k), generator=g, device="cuda", dtype=torch.int16)
    edge = round(500 * (1 - p_zero))
    return (r < edge).to(torch.int8).sub_((r >= 1000 - edge).to(torch.int8))


def _planes(g, n, k, p_zero):
    scale = lambda sigma: (torch.randn((n, k // GROUP), generator=g, device="cuda") * sigma).abs().half()  # noqa: E731
    return _trits(g, n, k, p_zero), _trits(g, n, k, p_zero), scale(0.02), scale(0.01)


def _x(g, *shape):
    return torch.randn(shape, generator=g, device="cuda").half()


def _blob(g, n, k, p_zero, fmt):
    return binding.ptqtp_pack(*_planes(g, n, k, p_zero), fmt=fmt)[0]


def _out(*shape):
    return torch.zeros(shape, dtype=torch.float16, device="cuda")


def _prepare_layer(case, g):
    h, kv, inter, m, fmt, form = (case[v] for v in ("hidden", "kv", "inter", "m", "fmt", "form"))
    shape = {"q": (h, h), "k": (kv, h), "v": (kv, h), "o": (h, h), "gate": (inter, h), "up": (inter, h), "down": (h, inter)}
    rows = (lambda n: (n,)) if m == 1 else (lambda n: (m, n))
    layers, outs = [], []
    ws = None
    if form == "ws":
        ws = torch.empty(max(binding.gemm_skinny_workspace_size(n, k, m, fmt=fmt) for n, k in shape.values()),
                         dtype=torch.uint8, device="cuda")
    for _ in range(case["layers"]):
        blob = {name: _blob(g, n, k, case["p_zero"], fmt) for name, (n, k) in shape.items()}
        y = {name: _out(*rows(n)) for name, (n, k) in shape.items() if form != "fused" or name != "up"}
        # q, k and v share their activations, and so do gate and up
        xs = {"q": _x(g, *rows(h)), "o": _x(g, *rows(h)), "gate": _x(g, *rows(h)), "down": _x(g, *rows(inter))}
        xs["k"] = xs["v"] = xs["q"]
        xs["up"] = xs["gate"]
        layers.append((blob, xs, y))
        outs.append(y)

    def step():
        for blob, xs, y in layers:
            if form == "fused":
                binding.ptqtp_gemv_multi([blob["q"], blob["k"], blob["v"]], [h, kv, kv], h, xs["q"], ys=[y["q"], y["k"], y["v"]])
                binding.ptqtp_gemv(blob["o"], h, h, y["q"], y=y["o"], fmt=fmt)
                binding.ptqtp_gemv_multi([blob["gate"], blob["up"]], [inter, inter], h, y["o"], ys=[y["gate"]],
                                         epilogue=binding.EPILOGUE_GATED_PAIR)
                binding.ptqtp_gemv(blob["down"], h, inter, y["gate"], y=y["down"], fmt=fmt)
                continue
            for name, (n, k) in shape.items():
                if form == "separate":
                    binding.ptqtp_gemv(blob[name], n, k, xs[name], y=y[name], fmt=fmt)
                elif form == "skinny":
                    binding.ptqtp_gemm_skinny(blob[name], n, k, xs[name], Y=y[name], fmt=fmt)
                else:
                    binding.ptqtp_gemm_skinny_ws(blob[name], n, k, xs[name], Y=y[name], workspace=ws, fmt=fmt)

    old = binding.ptqtp_set_overlap(case["level"])       # the level is part of what a graph captures
    try:
        step()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step()
    finally:
        binding.ptqtp_set_overlap(old)
    return {"case": case, "graph": graph, "layers": layers, "ws": ws, "out": outs}


def prepare(case, seed):
    g = _generator(seed)
    kind = case["kind"]
    if kind == "layer":
        return _prepare_layer(case, g)
    n, k, fmt = case["n"], case["k"], case["fmt"]
    if kind == "call":
        return {"case": case, "blob": _blob(g, n, k, 0.4, fmt), "x": _x(g, k), "y": _out(n)}
    if kind == "host":
        host = lambda t: t.cpu().pin_memory()  # noqa: E731
        return {"case": case, "blob": _blob(g, n, k, 0.4, fmt), "x": host(_x(g, k)), "y": host(_out(n)),
                "x_dev": _out(k), "y_dev": _out(n)}
    if kind == "pack":
        size = binding.packed_size(n, k, fmt=fmt)
        return {"case": case, "planes": _planes(g, n, k, 0.4), "blob": torch.empty(size, dtype=torch.uint8, device="cuda"),
                "status": torch.zeros(1, dtype=torch.int32, device="cuda")}
    if kind == "unpack":
        return {"case": case, "blob": _blob(g, n, k, 0.4, fmt)}
    return {"case": case, "w": make_weights_device(n, k, seed=seed)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "layer":
        state["graph"].replay()
        return state["out"]
    n, k, fmt = case["n"], case["k"], case["fmt"]
    if kind == "call":
        return binding.ptqtp_gemv(state["blob"], n, k, state["x"], y=state["y"], fmt=fmt)
    if kind == "host":
        y = binding.ptqtp_gemv_host(state["blob"], n, k, state["x"], state["y"], state["x_dev"], state["y_dev"], fmt=fmt)
        torch.cuda.current_stream().synchronize()        # the caller reads y
        return y
    if kind == "pack":
        return binding.ptqtp_pack(*state["planes"], packed=state["blob"], dev_status=state["status"], fmt=fmt)
    if kind == "unpack":
        return binding.ptqtp_unpack(state["blob"], n, k, fmt=fmt)
    t1, t2, a1, a2 = binding.ptqtp_decompose(state["w"])
    blob, status = binding.ptqtp_pack(t1, t2, a1, a2, fmt=fmt)
    return {"t1": t1, "t2": t2, "alpha1": a1, "alpha2": a2, "blob": blob, "status": status}


# ---- what a pass cannot do without ----

def _packed_bytes(n, k):
    return n * k // 2 + 4 * n * (k // GROUP)             # 2 bits per trit and plane, two fp16 scales per group


def _linear(n, k, m):
    # every trit of both planes is one multiply-add per row of activations
    return {"bytes": _packed_bytes(n, k) + 2 * m * (n + k), "flops": 4 * n * k * m}


def work(case):
    kind = case["kind"]
    if kind == "layer":
        h, kv, inter, m = case["hidden"], case["kv"], case["inter"], case["m"]
        parts = [_linear(h, h, m), _linear(2 * kv, h, m), _linear(h, h, m), _linear(2 * inter, h, m), _linear(h, inter, m)]
        # q, k and v share their activations; a gated pair writes one output
        extra = 2 * m * h + (2 * m * inter if case["form"] == "fused" else 0)
        return {"bytes": case["layers"] * (sum(p["bytes"] for p in parts) - extra),
                "flops": case["layers"] * sum(p["flops"] for p in parts)}
    n, k = case["n"], case["k"]
    if kind in ("call", "host"):
        return _linear(n, k, 1)
    planes = 2 * n * k + 4 * n * (k // GROUP)
    if kind in ("pack", "unpack"):
        return {"bytes": planes + _packed_bytes(n, k), "flops": 0}
    # the weights are read once, planes and blob written once; the sweeps themselves work on what is on the chip
    return {"bytes": 4 * n * k + planes + _packed_bytes(n, k), "flops": 0}


def tolerance(case):
    kind = case["kind"]
    if kind in ("pack", "unpack"):
        return "exact"
    if kind == "quantise":
        return "exact"                                   # specified bit for bit: every operation rounded on its own
    if case.get("form") == "fused":
        # the rounding of every result to fp16 is carried through the chain: 5.3e-4 against the chain in 64 bits,
        # single values up to 4e-3 (gated products)
        return {"rel": 2e-3, "max": 1.6e-2}
    # one rounding to fp16: 2.1e-4 against the product in 64 bits, single values up to 5.5e-4
    return {"rel": 8e-4, "max": 2.2e-3}
