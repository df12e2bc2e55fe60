"""What a program built on this library spends its GPU time on, as cases that can be timed and compared.

Decoding one token (every linear layer of a few decoder layers, batch 1), the same stack for 2..16 sequences at
once, the product on layers whose sizes the tiled layout does not cover, and the offline side: quantising fp16
weights, turning step-1 integers into a packed operand, and the search over partitions and scale factors.
Sizes are those of the OPT- and Llama-2-shaped stacks that the benchmark runs, and their neighbourhood.

A decode step is a CUDA graph of the library's calls, which is how the benchmark (and a serving loop) runs it; the
single product, the ragged product and the offline calls are issued directly.
"""
import math

import torch

from paper_2407_02891_b200 import binding as bq

ACTS = {"none": bq.ACT_NONE, "relu": bq.ACT_RELU, "gelu": bq.ACT_GELU, "silu": bq.ACT_SILU}


def listed():
    return [
        # one small projection, called on its own: launch and host latency
        {"name": "gemv_1024", "kind": "gemv", "N": 1024, "K": 1024, "q": 3, "group": 128},
        # OPT-6.7B-shaped decoder layers, bfloat16 activations, small scaling groups, bias / ReLU / residual fused
        {"name": "decode_4096_bf16_g64", "kind": "decode", "hidden": 4096, "ffn": 16384, "kv": 0, "layers": 2, "q": 3, "group": 64,
         "style": "bf16", "act": "relu"},
        # OPT-30B-shaped decoder layers, the benchmark's default workload: six plain products per layer
        {"name": "decode_7168", "kind": "decode", "hidden": 7168, "ffn": 28672, "kv": 0, "layers": 2, "q": 3, "group": 128,
         "style": "plain", "act": "none"},
        # OPT-66B-shaped decoder layers, two planes, one scale per row (the paper's granularity)
        {"name": "decode_9216_q2_row", "kind": "decode", "hidden": 9216, "ffn": 36864, "kv": 0, "layers": 2, "q": 2, "group": 0,
         "style": "plain", "act": "none"},
        # Llama-2-70B-shaped decoder layers (grouped-query attention, gated feed-forward block): projections of one
        # activation in one launch, residual additions fused
        {"name": "decode_8192_fused", "kind": "decode", "hidden": 8192, "ffn": 28672, "kv": 2048, "layers": 2, "q": 3, "group": 128,
         "style": "fused", "act": "none"},
        # the same layers for 2, 8 and 16 sequences at once
        {"name": "batch2_8192", "kind": "batch", "hidden": 8192, "ffn": 28672, "kv": 2048, "layers": 1, "q": 3, "group": 128, "B": 2},
        {"name": "batch8_8192", "kind": "batch", "hidden": 8192, "ffn": 28672, "kv": 2048, "layers": 1, "q": 3, "group": 128, "B": 8},
        {"name": "batch16_8192", "kind": "batch", "hidden": 8192, "ffn": 28672, "kv": 2048, "layers": 1, "q": 3, "group": 128, "B": 16},
        # a projection whose width is no multiple of the tiled layout's window of 512 (canonical layout)
        {"name": "ragged_4096x11008", "kind": "ragged", "N": 4096, "K": 11008, "q": 3, "group": 128, "B": 1},
        # fp16 weights of one projection -> packed operand
        {"name": "quantize_7168", "kind": "quantize", "N": 7168, "K": 7168, "q": 3, "group": 128, "n_bits": 4, "tiled": True, "ints": False},
        # step-1 integers of one projection (from a solver outside the library) -> merged codes -> packed operand
        {"name": "merge_pack_7168", "kind": "merge_pack", "N": 7168, "K": 7168, "q": 3, "group": 128, "n_bits": 4, "tiled": True},
        # search over all partitions of 5 bits into 3 planes and 8 scale factors on 128 calibration tokens
        {"name": "search_4096", "kind": "search", "N": 4096, "K": 4096, "q": 3, "group": 128, "n_bits": 5, "T": 128, "scales": 8},
    ]


def _log(rng, lo, hi, step):
    """A multiple of `step` between lo and hi, spread evenly over the logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step)) * step))


def draw(rng):
    kind = rng.choice(["gemv", "decode", "decode", "decode", "batch", "batch", "batch", "ragged", "quantize", "merge_pack", "search"])
    q = rng.choice([2, 3, 3, 4])
    if kind == "gemv":
        return {"kind": kind, "N": _log(rng, 256, 8192, 8), "K": _log(rng, 1024, 8192, 512), "q": q, "group": rng.choice([0, 32, 64, 128])}
    if kind in ("decode", "batch"):
        hidden = _log(rng, 1024, 8192, 512)
        ffn = min(28672, 512 * round(hidden * rng.uniform(2.0, 4.0) / 512))
        kv = rng.choice([0, 8 * rng.randint(hidden // 64, hidden // 16)])
        case = {"kind": kind, "hidden": hidden, "ffn": ffn, "kv": kv, "layers": 1, "q": q}
        if kind == "batch":
            return dict(case, group=rng.choice([0, 128, 128, 128]), B=rng.randint(2, 16))
        style = rng.choice(["plain", "fused", "bf16"])
        group = rng.choice([0, 128, 128]) if style == "fused" else rng.choice([0, 32, 64, 128, 128])
        return dict(case, group=group, style=style, act=rng.choice(["none", "relu", "gelu", "silu"]) if style != "plain" else "none")
    if kind == "ragged":
        group = rng.choice([0, 32, 64, 128])
        step = group or 32
        return {"kind": kind, "N": _log(rng, 256, 5120, 1), "K": _log(rng, 1024, 11008, step), "q": q, "group": group, "B": rng.choice([1, 1, 1, 2, 4])}
    if kind == "search":
        group = rng.choice([0, 64, 128])
        return {"kind": kind, "N": _log(rng, 512, 4096, 8), "K": _log(rng, 512, 4096, 128), "q": rng.choice([2, 3]), "group": group,
                "n_bits": rng.choice([4, 5]), "T": 16 * rng.randint(2, 16), "scales": rng.randint(1, 8)}
    tiled = rng.random() < 0.75
    group = rng.choice([0, 32, 64, 128, 128])
    case = {"kind": kind, "N": _log(rng, 512, 8192, 8), "K": _log(rng, 512, 8192, 512 if tiled else 128), "q": q, "group": group,
            "n_bits": rng.randint(q, 5), "tiled": tiled}
    return dict(case, ints=rng.random() < 0.3) if kind == "quantize" else case


def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _scales(N, K, q, group, g):
    """alpha [q, N, G], z [N, G]: the benchmark's distributions, drawn on the device."""
    G = 1 if group == 0 else K // group
    a0 = 0.01 + 0.04 * torch.rand((N, G), generator=g, device="cuda")
    rows = [a0] + [a0 * 2.0 ** -i * (0.8 + 0.4 * torch.rand((N, G), generator=g, device="cuda")) for i in range(1, q)]
    z = 0.01 * torch.randn((N, G), generator=g, device="cuda")
    return torch.stack(rows).half().contiguous(), z.half()


def _layer(N, K, q, group, layout, g):
    """A packed layer with random bits, as a program holds it after its offline preparation."""
    planes = torch.randint(-2 ** 31, 2 ** 31 - 1, (q * N * K // 32,), generator=g, device="cuda", dtype=torch.int32).view(torch.uint8)
    alpha, z = _scales(N, K, q, group, g)
    canonical = bq.desc(N, K, q, group, bq.LAYOUT_CANONICAL)
    if layout == bq.LAYOUT_CANONICAL:
        return bq.Layer(canonical, planes, alpha.reshape(-1), z.reshape(-1))
    d = canonical.with_layout(bq.LAYOUT_TILED)
    packed, a, zz = bq.empty_operands(d, "cuda")
    bq.repack(canonical, planes, alpha.reshape(-1), z.reshape(-1), d, packed, a, zz)
    return bq.Layer(d, packed, a, zz)


def _randn(n, g, dtype=torch.float16, scale=1.0):
    return (scale * torch.randn(n, generator=g, device="cuda")).to(dtype)


def _shapes(case):
    """(name, N, K) of the linear layers of one decoder layer: OPT (kv = 0), or Llama-2 with k and v stacked."""
    h, f, kv = case["hidden"], case["ffn"], case["kv"]
    if kv:
        return [("q", h, h), ("kv", kv, h), ("o", h, h), ("gate", f, h), ("up", f, h), ("down", h, f)]
    return [("q", h, h), ("k", h, h), ("v", h, h), ("o", h, h), ("fc1", f, h), ("fc2", h, f)]


def _stack(case, seed):
    """Layers, activations and outputs of a stack, and the token's calls captured in a CUDA graph."""
    g = _rng(seed)
    B, q, group = case.get("B", 1), case["q"], case["group"]
    style = case.get("style", "plain")
    dtype = torch.bfloat16 if style == "bf16" else torch.float16
    x = {K: _randn(B * K, g, dtype) for K in (case["hidden"], case["ffn"])}
    workspaces, calls, keep, ys = {}, [], [], []

    def workspace(d):
        if (d.N, d.K) not in workspaces:
            workspaces[d.N, d.K] = bq.new_workspace(d, B)
        return workspaces[d.N, d.K]

    for _ in range(case["layers"]):
        layers = {n: _layer(N, K, q, group, bq.LAYOUT_TILED, g) for n, N, K in _shapes(case)}
        out = {n: torch.empty(B * L.d.N, dtype=dtype, device="cuda") for n, L in layers.items()}
        keep.append(layers)
        ys.append(out)
        if style == "plain":
            for n, L in layers.items():
                if B == 1:
                    calls.append(lambda L=L, y=out[n]: bq.gemv(L.d, L.packed, L.alpha, L.z, x[L.d.K], y, workspace(L.d)))
                else:
                    calls.append(lambda L=L, y=out[n]: bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, x[L.d.K], y, B, workspace(L.d)))
            continue
        # bias and activation follow the wide product, the residual the two that return to the hidden width
        act = ACTS[case["act"]]
        follow = {n: dict(bias=_randn(L.d.N, g, dtype, 0.1), residual=None, activation=act) if n in ("fc1", "up") else
                  dict(bias=None, residual=_randn(L.d.N, g, dtype), activation=bq.ACT_NONE) if n in ("o", "fc2", "down") else {}
                  for n, L in layers.items()}
        if style == "bf16":
            for n, L in layers.items():
                calls.append(lambda L=L, y=out[n], e=follow[n]: bq.gemv_bf16(L.d, L.packed, L.alpha, L.z, x[L.d.K], y, workspace=workspace(L.d), **e))
            continue
        together = [("q", "kv"), ("o",), ("gate", "up"), ("down",)] if case["kv"] else [("q", "k", "v"), ("o",), ("fc1",), ("fc2",)]
        for names in together:
            Ls = [layers[n] for n in names]
            if len(names) == 1:
                calls.append(lambda L=Ls[0], y=out[names[0]], e=follow[names[0]]:
                             bq.gemv_fused(L.d, L.packed, L.alpha, L.z, x[L.d.K], y, workspace=workspace(L.d), **e))
            else:
                d = bq.desc(sum(L.d.N for L in Ls), Ls[0].d.K, q, group, bq.LAYOUT_TILED)
                calls.append(lambda d=d, Ls=Ls, o=[out[n] for n in names]: bq.gemv_multi(d, Ls, x[d.K], o, workspace(d)))

    def token():
        for call in calls:
            call()

    token()   # workspaces exist and the kernels are loaded before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        token()
    return {"graph": graph, "out": ys, "keep": (keep, calls, x, workspaces)}


def _bit_to_plane(n_bits, q):
    """The lowest bits share a plane (a partition the search often picks)."""
    return [max(0, i - (n_bits - q)) for i in range(n_bits)]


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("decode", "batch"):
        return dict(_stack(case, seed), kind="stack")
    g = _rng(seed)
    N, K, q, group = case["N"], case["K"], case["q"], case["group"]
    G = 1 if group == 0 else K // group
    if kind in ("gemv", "ragged"):
        L = _layer(N, K, q, group, bq.LAYOUT_TILED if kind == "gemv" else bq.LAYOUT_CANONICAL, g)
        B = case.get("B", 1)
        return {"kind": "product", "L": L, "B": B, "x": _randn(B * K, g), "y": torch.empty(B * N, dtype=torch.float16, device="cuda"),
                "ws": bq.new_workspace(L.d, B)}
    d = bq.desc(N, K, q, group, bq.LAYOUT_TILED if case.get("tiled") else bq.LAYOUT_CANONICAL)
    half = lambda n: torch.empty(n, dtype=torch.float16, device="cuda")
    if kind == "quantize":
        packed, a, z = bq.empty_operands(d, "cuda")
        return {"kind": kind, "d": d, "W": _randn(N * K, g, scale=0.05), "n_bits": case["n_bits"], "b2p": _bit_to_plane(case["n_bits"], q),
                "out": (half(N * G), half(N * G), torch.empty(N * K, dtype=torch.uint8, device="cuda") if case["ints"] else None, packed, a, z)}
    if kind == "merge_pack":
        n_bits = case["n_bits"]
        packed, a, z = bq.empty_operands(d, "cuda")
        return {"kind": kind, "d": d, "n_bits": n_bits, "b2p": _bit_to_plane(n_bits, q),
                "w_int": torch.randint(0, 2 ** n_bits, (N * K,), generator=g, device="cuda", dtype=torch.uint8),
                "S": (0.002 + 0.03 * torch.rand(N * G, generator=g, device="cuda")).half(), "qbias": _randn(N * G, g, scale=0.1),
                "codes": torch.empty(N * K, dtype=torch.uint8, device="cuda"), "alpha": half(q * N * G), "z": half(N * G), "out": (packed, a, z)}
    return {"kind": "search", "args": (N, K, q, group, _randn(N * K, g, scale=0.05).view(N, K), _randn(case["T"] * K, g).view(case["T"], K),
                                       case["n_bits"], bq.partitions(case["n_bits"], q), bq.reexplore_factors(case["n_bits"], case["scales"]))}


def run(state):
    kind = state["kind"]
    if kind == "stack":
        state["graph"].replay()
        return state["out"]
    if kind == "product":
        L, B = state["L"], state["B"]
        if B == 1:
            bq.gemv(L.d, L.packed, L.alpha, L.z, state["x"], state["y"], state["ws"])
        else:
            bq.gemm_smallbatch(L.d, L.packed, L.alpha, L.z, state["x"], state["y"], B, state["ws"])
        return state["y"]
    if kind == "quantize":
        S, qbias, w_int, packed, alpha, z = state["out"]
        bq.quantize_rtn(state["d"], state["W"], state["n_bits"], state["b2p"], S, qbias, w_int, packed, alpha, z)
        return [t for t in state["out"] if t is not None]
    if kind == "merge_pack":
        bq.merge_linear(state["d"], state["w_int"], state["S"], state["qbias"], state["n_bits"], state["b2p"], state["codes"], state["alpha"], state["z"])
        bq.pack(state["d"], state["codes"], state["alpha"], state["z"], *state["out"])
        return [state["codes"], state["alpha"], state["z"]] + [t for t in state["out"] if t is not None]
    err, rows, _ = bq.grid_search(*state["args"])
    return [err, rows]   # the chosen index is left out: two candidates closer than the tolerance may swap places


def _operand_bytes(N, K, q, group):
    G = 1 if group == 0 else K // group
    return q * N * K // 8 + 2 * (q + 1) * N * G


def work(case):
    kind = case["kind"]
    if kind in ("decode", "batch"):
        B, layers = case.get("B", 1), case["layers"]
        shapes = _shapes(case)
        bytes_ = sum(_operand_bytes(N, K, case["q"], case["group"]) + 2 * B * N for _, N, K in shapes) * layers + 2 * B * (case["hidden"] + case["ffn"])
        if case.get("style", "plain") != "plain":
            bytes_ += 2 * (2 * case["hidden"] + case["ffn"]) * layers
        return {"bytes": bytes_, "flops": sum(2 * B * N * K for _, N, K in shapes) * layers}
    N, K, q, group = case["N"], case["K"], case["q"], case["group"]
    G = 1 if group == 0 else K // group
    operand = _operand_bytes(N, K, q, group)
    if kind in ("gemv", "ragged"):
        B = case.get("B", 1)
        return {"bytes": operand + 2 * B * (N + K), "flops": 2 * B * N * K}
    if kind == "quantize":
        return {"bytes": 2 * N * K + operand + 4 * N * G + (N * K if case["ints"] else 0), "flops": 0}
    if kind == "merge_pack":   # integers in; codes, planes, and both arrangements of the scales out
        return {"bytes": 2 * N * K + 4 * N * G + operand + 2 * (q + 1) * N * G, "flops": 0}
    P = bq.lib().bcq_partition_count(case["n_bits"], q)
    S, T = case["scales"], case["T"]
    return {"bytes": 2 * N * K + 2 * T * K + 4 * S * P * N + 8 * S * P, "flops": 2.0 * N * K * T * P * S}


def tolerance(case):
    """About four times what the paths were measured to differ from an fp64 evaluation (rel 2.1e-4 for one rounding to
    fp16, 3.0e-4 where fp16 table entries come before it; bfloat16 rounds eight times coarser)."""
    kind = case["kind"]
    if kind in ("quantize", "merge_pack"):
        return "exact"
    if kind == "search":
        return {"rel": 3e-4, "max": 2e-3}   # fp16 differences of weights, fp32 sums of squares: 4e-5 .. 8e-5 measured
    if case.get("style") == "bf16":
        return {"rel": 7e-3, "max": 1.2e-2}
    return {"rel": 1.2e-3, "max": 6e-3}
