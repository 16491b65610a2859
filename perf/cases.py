"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is a dict of plain values with a "kind":

    linear    one cq_gemm: N x K weights of B bits in groups of G, M rows of activations
    layer     the four linears of a transformer layer, one cq_gemm each, in the order a forward pass runs them:
              qkv (hidden -> N_qkv), o (hidden -> hidden), gate_up (hidden -> 2 I), down (I -> hidden)
    sweep     one cq_gemm for every (B, G) of the bit-width / group-size sweep, one matrix size
    mlp       cq_mlp_swiglu: gate_up, gated activation and quantiser, down
    routed    cq_gemm_routed: T tokens, `top` routes each, over E matrices with uneven loads
    quantise  cq_encode, cq_pack_codes, cq_repack, cq_unpack: a trained fp32 matrix to the device layout and back to a checkpoint

"mode" is the activation mode ("model": the model dtype, "a8": Dynamic A8) and "dtype" the model dtype ("bf16", "f16").
Sizes are those of this repository's configurations and benchmark (4096 and 8192 square, the Llama-3-8B linears,
the Llama-3-70B MLP), and generic ones in between.
"""
import torch

import paper_2608_06763_b200 as cq

SWEEP = [(B, G) for B in (1, 2, 3, 4, 6, 8) for G in (32, 64, 128)]
LAYER = {"hidden": 4096, "n_qkv": 6144, "inter": 14336}   # the Llama-3-8B linears
MODE = {"model": cq.CQ_MODEL_DTYPE, "a8": cq.CQ_DYN_A8}
DTYPE = {"bf16": torch.bfloat16, "f16": torch.float16}


def listed():
    return [
        # one small projection for one token: the shortest call there is, launch and latency
        {"name": "linear 4096 w4 m1", "kind": "linear", "N": 4096, "K": 4096, "B": 4, "G": 128, "M": 1, "mode": "model", "dtype": "bf16"},
        # every format a checkpoint can be stored in, one token: the benchmark's headline sweep
        {"name": "sweep 8192 m1", "kind": "sweep", "N": 8192, "K": 8192, "M": 1, "mode": "model", "dtype": "bf16"},
        # single-stream decoding: a layer's linears for one token
        {"name": "decode layer w4 m1", "kind": "layer", **LAYER, "B": 4, "G": 128, "M": 1, "mode": "model", "dtype": "bf16"},
        # batched decoding, an odd batch
        {"name": "decode layer w4 m13", "kind": "layer", **LAYER, "B": 4, "G": 128, "M": 13, "mode": "model", "dtype": "bf16"},
        # batched decoding through the fused MLP block with INT8 activations on both sides
        {"name": "decode mlp w4 a8 m16", "kind": "mlp", "hidden": 4096, "inter": 14336, "B": 4, "G": 128, "M": 16, "mode": "a8", "dtype": "bf16"},
        # a large decoding batch with INT8 activations, eight-bit weights
        {"name": "decode layer w8 a8 m64", "kind": "layer", **LAYER, "B": 8, "G": 128, "M": 64, "mode": "a8", "dtype": "bf16"},
        # a short prompt of ragged length, binary16 model
        {"name": "prefill layer w4 f16 m200", "kind": "layer", **LAYER, "B": 4, "G": 128, "M": 200, "mode": "model", "dtype": "f16"},
        # an ordinary prompt
        {"name": "prefill layer w4 m1024", "kind": "layer", **LAYER, "B": 4, "G": 128, "M": 1024, "mode": "model", "dtype": "bf16"},
        # a mixture-of-experts projection: few rows for each of many matrices
        {"name": "routed w4 e16 t192", "kind": "routed", "E": 16, "N": 2816, "K": 2048, "B": 4, "G": 64, "T": 192, "top": 2, "mode": "model", "dtype": "bf16"},
        # the largest prefill products, three-bit weights in the model dtype and four-bit ones in Dynamic A8
        {"name": "prefill 70b gate_up w3 m4096", "kind": "linear", "N": 57344, "K": 8192, "B": 3, "G": 128, "M": 4096, "mode": "model", "dtype": "bf16"},
        {"name": "prefill 70b down w4 a8 m4096", "kind": "linear", "N": 8192, "K": 28672, "B": 4, "G": 128, "M": 4096, "mode": "a8", "dtype": "bf16"},
        # quantising a trained matrix under the dual-path objective, once for each matrix of a model
        {"name": "quantise 2048x4096 w4", "kind": "quantise", "N": 2048, "K": 4096, "B": 4, "G": 128, "objective": "joint", "effort": "fast"},
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], evenly spread over the logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def _multiple(rng, lo, hi, of):
    return max(of, _log(rng, lo, hi) // of * of)


def draw(rng):
    fmt = {"B": rng.choice([2, 3, 4, 4, 4, 5, 6, 8]), "G": rng.choice([32, 64, 128, 128, 256])}
    how = {"mode": rng.choice(["model", "model", "a8"]), "dtype": rng.choice(["bf16", "bf16", "f16"])}
    kind = rng.choice(["linear", "linear", "linear", "layer", "layer", "sweep", "mlp", "routed", "quantise"])
    G = fmt["G"]
    if kind == "linear":
        M, G = _log(rng, 1, 4096), rng.choice([G, G, 512])
        fmt["G"] = G
        K = _multiple(rng, 1024, 28672, G)
        N = _log(rng, 1024, 57344)
        while N * K > 470e6:
            N //= 2
        if rng.random() < 0.6:
            N = N // 8 * 8
        return {"kind": kind, "N": N, "K": K, **fmt, "M": M, **how}
    if kind == "layer":
        hidden = _multiple(rng, 1024, 4096, 256)
        return {"kind": kind, "hidden": hidden, "n_qkv": hidden + 2 * _multiple(rng, hidden // 8, hidden // 2, 64), "inter": _multiple(rng, 2 * hidden, 4 * hidden, 256),
                **fmt, "M": _log(rng, 1, 1024), **how}
    if kind == "sweep":
        return {"kind": kind, "N": _log(rng, 1024, 8192) // 8 * 8, "K": _multiple(rng, 1024, 8192, 128), "M": rng.choice([1, 1, 2, 3, 4]), **how}
    if kind == "mlp":
        return {"kind": kind, "hidden": _multiple(rng, 1024, 4096, 256), "inter": _multiple(rng, 2048, 14336, 256), **fmt, "M": _log(rng, 1, 1024), **how}
    if kind == "routed":
        return {"kind": kind, "E": rng.choice([8, 16, 32]), "N": _log(rng, 1024, 4096) // 8 * 8, "K": _multiple(rng, 1024, 4096, 256), **fmt,
                "T": _log(rng, 16, 1024), "top": rng.choice([1, 2, 4]), **how}
    return {"kind": kind, "N": _log(rng, 256, 2048), "K": _multiple(rng, 1024, 4096, G), "B": rng.choice([3, 4, 4, 5]), "G": G,
            "objective": rng.choice(["joint", "continuous"]), "effort": "fast"}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + 12345)
    return g


def _laplace(shape, g, scale):
    d = (torch.rand(shape, generator=g, device="cuda") - 0.5).clamp_(-0.4999999, 0.4999999)
    return -scale * torch.sign(d) * torch.log1p(-2.0 * d.abs())


def _matrix(g, N, K, B, G):
    """A stored matrix: bell-shaped signed codes as a fit leaves them, shape parameters of monotone cubics."""
    top = 1 if B == 1 else (1 << (B - 1)) - 1
    codes = torch.empty((N, K), dtype=torch.int8, device="cuda")
    rows = max(1, (1 << 26) // K)
    for r in range(0, N, rows):
        n = min(rows, N - r)
        if B == 1:
            codes[r:r + n] = torch.where(torch.rand((n, K), generator=g, device="cuda") < 0.5, -1, 1)
        else:
            codes[r:r + n] = _laplace((n, K), g, 0.22 * top + 0.35).round_().clamp_(-top, top)
    shape = (N, K // G)
    s = 0.03 + 0.06 * torch.rand(shape, generator=g, device="cuda")
    a = (0.5 + 0.5 * torch.rand(shape, generator=g, device="cuda")).half()
    b = (-0.3 * torch.rand(shape, generator=g, device="cuda")).half()
    return codes, s, a, b


def _packed(g, N, K, B, G):
    codes, s, a, b = _matrix(g, N, K, B, G)
    return cq.cq_repack(cq.cq_pack_codes(codes, B), s, a, b, B, G, N, K)


def _activations(g, M, K, dtype):
    """N(0, 1) with one column in a hundred twenty times larger, as activations of a trained model look."""
    x = torch.randn((M, K), generator=g, device="cuda")
    x[:, torch.randperm(K, generator=g, device="cuda")[: K // 100]] *= 20.0
    return x.to(DTYPE[dtype])


def _product(g, c, N, K, B=None, G=None):
    """One linear with what a serving program keeps for it: weights, input, output, workspace."""
    B, G, M, mode = B or c["B"], G or c["G"], c["M"], MODE[c["mode"]]
    pw = _packed(g, N, K, B, G)
    x = _activations(g, M, K, c["dtype"])
    ws = torch.zeros(cq.cq_workspace_bytes(B, G, M, N, K, mode), dtype=torch.uint8, device="cuda")
    return pw, x, mode, ws, torch.empty((M, N), dtype=x.dtype, device="cuda")


def _routes(g, c):
    load = torch.rand((c["T"], c["E"]), generator=g, device="cuda") + 0.5 * torch.rand(c["E"], generator=g, device="cuda")   # some matrices are preferred
    chosen = load.topk(c["top"], dim=1).indices
    return chosen, chosen.flatten().argsort(stable=True)


def _layer_sizes(c):
    return [(c["n_qkv"], c["hidden"]), (c["hidden"], c["hidden"]), (2 * c["inter"], c["hidden"]), (c["hidden"], c["inter"])]


def prepare(case, seed):
    c, g = case, _generator(seed)
    kind = c["kind"]
    if kind == "linear":
        return {"kind": kind, "products": [_product(g, c, c["N"], c["K"])]}
    if kind == "layer":
        return {"kind": kind, "products": [_product(g, c, N, K) for N, K in _layer_sizes(c)]}
    if kind == "sweep":
        return {"kind": kind, "products": [_product(g, c, c["N"], c["K"], B, G) for B, G in SWEEP]}
    if kind == "mlp":
        H, I, M = c["hidden"], c["inter"], c["M"]
        up, down = _packed(g, 2 * I, H, c["B"], c["G"]), _packed(g, H, I, c["B"], c["G"])
        x = _activations(g, M, H, c["dtype"])
        need = cq.lib().cq_mlp_workspace_bytes(c["B"], c["G"], c["B"], c["G"], M, H, I, H, MODE[c["mode"]])
        return {"kind": kind, "up": up, "down": down, "x": x, "mode": MODE[c["mode"]],
                "ws": torch.zeros(need, dtype=torch.uint8, device="cuda"), "y": torch.empty((M, H), dtype=x.dtype, device="cuda")}
    if kind == "routed":
        E, T = c["E"], c["T"]
        experts = [_packed(g, c["N"], c["K"], c["B"], c["G"]) for _ in range(E)]
        x = _activations(g, T, c["K"], c["dtype"])
        chosen, order = _routes(g, c)
        counts = torch.bincount(chosen.flatten(), minlength=E).cumsum(0).tolist()
        return {"kind": kind, "experts": experts, "x": x, "route_token": (order // c["top"]).to(torch.int32), "offset": [0] + counts, "mode": MODE[c["mode"]]}
    W = torch.randn((c["N"], c["K"]), generator=g, device="cuda") * 0.02
    W = torch.where(torch.rand(W.shape, generator=g, device="cuda") < 0.001, 10.0 * W, W)   # a few outliers
    return {"kind": kind, "W": W, "B": c["B"], "G": c["G"], "objective": cq.CQ_FIT_JOINT if c["objective"] == "joint" else cq.CQ_FIT_CONTINUOUS, "effort": c["effort"]}


def run(state):
    kind = state["kind"]
    if kind in ("linear", "layer", "sweep"):
        return [cq.cq_gemm(pw, x, mode, ws, y) for pw, x, mode, ws, y in state["products"]]
    if kind == "mlp":
        return cq.cq_mlp_swiglu(state["up"], state["down"], state["x"], state["mode"], state["ws"], state["y"])
    if kind == "routed":
        return cq.cq_gemm_routed(state["experts"], state["x"], state["route_token"], state["offset"], state["mode"])
    W, B, G = state["W"], state["B"], state["G"]
    codes, s, a, b = cq.cq_encode(W, B, G, state["objective"], state["effort"])
    packed = cq.cq_pack_codes(codes, B)
    pw = cq.cq_repack(packed, s, a, b, B, G, *W.shape)
    return {"codes": codes, "packed": packed, "scale": s, "a": a, "b": b, "stored": cq.cq_unpack(pw)}   # read back: the device layout itself is private


# ------------------------------------------------------------------ what a pass cannot do without, and what it may differ by
def _linear_work(M, N, K, B, G):
    return N * K * (B / 8 + 8 / G) + 2 * M * (K + N), 2.0 * M * N * K


def work(case):
    c, kind = case, case["kind"]
    if kind == "linear":
        parts = [_linear_work(c["M"], c["N"], c["K"], c["B"], c["G"])]
    elif kind == "layer":
        parts = [_linear_work(c["M"], N, K, c["B"], c["G"]) for N, K in _layer_sizes(c)]
    elif kind == "sweep":
        parts = [_linear_work(c["M"], c["N"], c["K"], B, G) for B, G in SWEEP]
    elif kind == "mlp":
        H, I, M = c["hidden"], c["inter"], c["M"]
        parts = [_linear_work(M, 2 * I, H, c["B"], c["G"]), _linear_work(M, H, I, c["B"], c["G"])]
        parts.append((-2 * M * 3 * I, 0.0))   # the intermediate is neither an input nor an output
    elif kind == "routed":
        R = c["T"] * c["top"]
        parts = [(c["E"] * c["N"] * c["K"] * (c["B"] / 8 + 8 / c["G"]) + 2 * c["T"] * c["K"] + 2 * R * c["N"], 2.0 * R * c["N"] * c["K"])]
    else:
        # 4 bytes in, a code of one byte and the two packed forms out, for each weight; the search assigns every weight
        # about 550 times (candidates x rounds), some eight operations each, and twice that under the joint objective
        n = c["N"] * c["K"]
        parts = [(n * (4 + 1 + 2 * c["B"] / 8) + 16 * n / c["G"], n * 4400.0 * (2 if c["objective"] == "joint" else 1))]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    if case["kind"] == "quantise":
        return "exact"   # the search takes its decisions in fp64 in a fixed order: every byte is determined
    if case["kind"] == "mlp":
        # differences of 1e-3 in the first product move activations across INT8 rounding boundaries: whole steps of max|act| / 127
        return {"rel": 2e-2, "max": 0.2}
    return {"rel": 1e-2, "max": 0.05}   # bf16 outputs and temporary operands: 2^-9 each


# ------------------------------------------------------------------ the same results in 64 bits
def _levels(codes, a, b, B, G):
    """sign(k) q(|k| / M) of rows of codes, q(t) = t (a + t (b + c t)) with c = 1 - a - b; two bits and fewer have no shape."""
    k = codes.double()
    if B <= 2:
        return k
    t = k.abs() / ((1 << (B - 1)) - 1)
    a, b = (v.double().repeat_interleave(G, dim=1) for v in (a, b))
    return k.sign() * t * (a + t * (b + t * (1.0 - a - b)))


def _carriers(codes, a, b, B, G):
    """sign(k) RNE(127 q), q by the 32-bit sequence that the format prescribes (a fused product and sum rounds once)."""
    k = codes.double()
    if B <= 2:
        return 127.0 * k
    a, b = (v.float().repeat_interleave(G, dim=1) for v in (a, b))
    c = ((1.0 - a) - b).double()
    t = (codes.float().abs() / float((1 << (B - 1)) - 1))
    t64 = t.double()
    q = t * (t64 * (t64 * c + b.double()).float().double() + a.double()).float()
    return k.sign() * (127.0 * q).round().clamp(0, 127).double()


def _exact_product(matrix, x, B, G, mode):
    """x W^T in 64 bits; for Dynamic A8 from the INT8 activations and carriers, which the format defines in 32 bits."""
    codes, s, a, b = matrix
    out = torch.empty((x.shape[0], codes.shape[0]), dtype=torch.float64, device="cuda")
    if mode == "a8":
        f = x.float()
        d = f.abs().amax(dim=1, keepdim=True).clamp_min(1e-10) / 127.0
        v = f / d
        x64 = (v.sign() * (v.double().abs() + 0.5).floor()).clamp(-127, 127).double()
        decode, last = _carriers, d.double() / 127.0
    else:
        x64, decode, last = x.double(), _levels, 1.0
    rows = max(1, (1 << 25) // codes.shape[1])
    for r in range(0, codes.shape[0], rows):
        part = slice(r, r + rows)
        w = decode(codes[part], a[part], b[part], B, G) * s[part].double().repeat_interleave(G, dim=1)
        out[:, part] = x64 @ w.T * last
    return out


def exact(case, seed):
    c, g, kind = case, _generator(seed), case["kind"]
    if kind in ("linear", "layer", "sweep"):
        sizes = {"linear": lambda: [(c["N"], c["K"])], "layer": lambda: _layer_sizes(c), "sweep": lambda: [(c["N"], c["K"])] * len(SWEEP)}[kind]()
        out = []
        for (N, K), (B, G) in zip(sizes, SWEEP if kind == "sweep" else [(c["B"], c["G"])] * len(sizes)):
            m = _matrix(g, N, K, B, G)
            out.append(_exact_product(m, _activations(g, c["M"], K, c["dtype"]), B, G, c["mode"]))
        return out
    if kind == "mlp":
        H, I = c["hidden"], c["inter"]
        up, down = _matrix(g, 2 * I, H, c["B"], c["G"]), _matrix(g, H, I, c["B"], c["G"])
        # both operators in front return the model dtype, and the last one quantises what it is given
        h = _exact_product(up, _activations(g, c["M"], H, c["dtype"]), c["B"], c["G"], c["mode"]).to(DTYPE[c["dtype"]]).double()
        act = (torch.nn.functional.silu(h[:, :I]) * h[:, I:]).to(DTYPE[c["dtype"]])
        return _exact_product(down, act, c["B"], c["G"], "a8")
    if kind == "routed":
        experts = [_matrix(g, c["N"], c["K"], c["B"], c["G"]) for _ in range(c["E"])]
        x = _activations(g, c["T"], c["K"], c["dtype"])
        chosen, order = _routes(g, c)
        expert, token = chosen.flatten()[order], order // c["top"]
        out = torch.empty((order.numel(), c["N"]), dtype=torch.float64, device="cuda")
        for e in range(c["E"]):
            mine = expert == e
            out[mine] = _exact_product(experts[e], x[token[mine]], c["B"], c["G"], c["mode"])
        return out
    return None   # codes and bytes: compared as they are
