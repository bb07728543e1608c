"""The work that a user of the library has it do, as cases that can be timed and compared.

A model is brought in once ("encode": quantize the FP16 weights to power-of-two codes, put codes and scales into the
kernels' order), its weights are unpacked to 16-bit matrices where another kernel wants them ("dequant"), and it is served:
one token at a time ("decode": the projections of several decoder layers, recorded in a CUDA graph; "gemv": one eager call),
for small batches and for prompts ("gemm").  Shapes are those of the repository's workloads and tests (4096 .. 28672 wide
projections, 2 / 3 / 4 bits, groups of 64 and 128, FP16 and BF16), with ragged token counts and odd row counts beside them;
codes are tiled (the layout that serving uses) or canonical (the interchange layout: the default of the binding, and the only
one that takes row counts that are no multiple of 16).
"""
from __future__ import annotations

import torch

from paper_2507_11959_b200 import binding as B

LARGEST = 28672 * 8192       # weights of the largest single matrix
LARGEST_SHORT = 4096 * 11008  # ... and of the largest one that is encoded, or multiplied as it came


def listed() -> list[dict]:
    return [
        # one eager GEMV on the smallest projection: launch and call overhead count as much as bandwidth
        dict(name="gemv_4096x4096_3bit", op="gemv", n=4096, k=4096, bits=3, group=128, dtype="f16", layout="tiled"),
        # one decode token through eight decoder layers: five projections each, replayed as a CUDA graph
        dict(name="decode_8_layers_3bit", op="decode", layers=8, hidden=4096, ffn=11008, bits=3, group=128),
        # the largest projection for one token, with the other activation type, width and group
        dict(name="gemv_28672x8192_4bit_bf16", op="gemv", n=28672, k=8192, bits=4, group=64, dtype="bf16", layout="tiled"),
        # codes as they come (no repacking), a row count that is not a multiple of anything
        dict(name="gemv_canonical_10007x4096_2bit", op="gemv", n=10007, k=4096, bits=2, group=128, dtype="f16", layout="canonical"),
        # a decode batch of four requests on the widest projection of a 5120-wide model
        dict(name="gemm_4_tokens_15360x5120", op="gemm", m=4, n=15360, k=5120, bits=3, group=128, dtype="f16", layout="tiled"),
        # a decode batch of 32 requests on its narrowest, deepest one
        dict(name="gemm_32_tokens_5120x13824", op="gemm", m=32, n=5120, k=13824, bits=3, group=128, dtype="f16", layout="tiled"),
        # a short prompt: ragged token count, ragged rows, BF16, small groups
        dict(name="gemm_301_tokens_11024x4096_bf16", op="gemm", m=301, n=11024, k=4096, bits=4, group=64, dtype="bf16", layout="tiled"),
        # a long prompt on the largest projection
        dict(name="gemm_2048_tokens_28672x8192", op="gemm", m=2048, n=28672, k=8192, bits=3, group=128, dtype="f16", layout="tiled"),
        # a batch on codes as they come, odd row count
        dict(name="gemm_canonical_200_tokens_4099x11008", op="gemm", m=200, n=4099, k=11008, bits=3, group=128, dtype="f16", layout="canonical"),
        # unpacking a small projection, and a large one
        dict(name="dequant_4096x4096_2bit", op="dequant", n=4096, k=4096, bits=2, group=64, dtype="f16"),
        dict(name="dequant_28672x8192_3bit_bf16", op="dequant", n=28672, k=8192, bits=3, group=128, dtype="bf16"),
        # bringing in one projection with the published scale search (200 candidates per group)
        dict(name="encode_search_11008x4096_3bit", op="encode", n=11008, k=4096, bits=3, group=128, rule="search"),
    ]


def _spread(rng, low: int, high: int, step: int = 1) -> int:
    """A multiple of `step` in [low, high], spread evenly over its logarithm."""
    v = low * (high / low) ** rng.random()
    return max(low, min(high, int(v / step + 0.5) * step))


def draw(rng) -> dict:
    op = rng.choice(("gemv", "decode", "gemm", "gemm", "dequant", "encode"))
    bits, group = rng.choice((2, 3, 4)), rng.choice((64, 128))
    dtype = rng.choice(("f16", "bf16"))
    if op == "decode":
        hidden = _spread(rng, 1024, 4096, 128)
        return dict(op=op, layers=rng.randint(2, 8), hidden=hidden, ffn=_spread(rng, 2 * hidden, int(2.6875 * hidden), 128), bits=bits, group=group)
    k = _spread(rng, 1024, 28672, 128)
    layout = rng.choice(("tiled", "tiled", "tiled", "canonical")) if op in ("gemv", "gemm") else None
    top = LARGEST_SHORT if op == "encode" or layout == "canonical" else LARGEST
    n = _spread(rng, 1024, min(28672, top // k // 16 * 16), 16 if op == "encode" or layout == "tiled" else 1)
    case = dict(op=op, n=n, k=k, bits=bits, group=group)
    if op == "encode":
        return dict(case, rule=rng.choice(("top", "paper", "search", "search")))
    case["dtype"] = dtype
    if op == "dequant":
        return case
    if op == "gemm":
        case["m"] = _spread(rng, 2, 2048)
    return dict(case, layout=layout)


_DTYPE = {"f16": torch.float16, "bf16": torch.bfloat16}
_RULE = {"top": B.SCALE_TOP, "paper": B.SCALE_PAPER_S0, "search": B.SCALE_SEARCH}


def _weights(n: int, k: int, gen: torch.Generator) -> torch.Tensor:
    """[n, k] FP16, Student-t(5) * 0.02: bell-shaped with heavy tails, as projection weights are."""
    w = torch.randn(n, k, generator=gen, device="cuda")
    chi2 = torch.zeros_like(w)
    for _ in range(5):
        z = torch.randn(n, k, generator=gen, device="cuda")
        chi2.addcmul_(z, z)
    return w.div_(chi2.div_(5.0).sqrt_()).mul_(0.02).to(torch.float16)


def _activations(m: int, k: int, dtype: str, gen: torch.Generator) -> torch.Tensor:
    """[m, k] ~ N(0, 1) with 1 % of the channels (the same ones for every token) twenty times as large."""
    x = torch.randn(m, k, generator=gen, device="cuda")
    x[:, torch.randperm(k, generator=gen, device="cuda")[: k // 100]] *= 20.0
    return x.to(_DTYPE[dtype])


def _codes(n: int, k: int, bits: int, group: int, layout: str, gen: torch.Generator):
    packed, scales = B.pot_quantize_ref(_weights(n, k, gen), bits, group, B.SCALE_TOP)
    if layout == "tiled":
        packed, scales = B.pot_repack(packed, k, bits, 0), B.pot_repack_scales(scales, k, group, 0)
    return packed, scales


def prepare(case: dict, seed: int) -> dict:
    gen = torch.Generator(device="cuda").manual_seed(seed)
    op, bits, group = case["op"], case["bits"], case["group"]
    state = dict(case)
    if op == "decode":
        h, f = case["hidden"], case["ffn"]
        calls = []
        for _ in range(case["layers"]):
            for n, k in ((3 * h, h), (h, h), (f, h), (f, h), (h, f)):  # qkv, o, gate, up, down
                packed, scales = _codes(n, k, bits, group, "tiled", gen)
                calls.append((packed, scales, k, _activations(1, k, "f16", gen)[0], torch.empty(n, dtype=torch.float16, device="cuda"),
                              B.new_workspace(B.pot_gemv_workspace_bytes(n, k, bits, group))))

        def token():
            for packed, scales, k, x, y, ws in calls:
                B.pot_gemv(packed, scales, k, bits, group, x, B.TILED, y=y, workspace=ws)

        graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(stream):
            token()  # once outside of the capture
            with torch.cuda.graph(graph, stream=stream):
                token()
        torch.cuda.current_stream().wait_stream(stream)
        state.update(calls=calls, graph=graph, ys=[c[4] for c in calls])
        return state
    n, k = case["n"], case["k"]
    if op == "encode":
        state["w"] = _weights(n, k, gen)
        return state
    if op == "dequant":
        state["packed"], state["scales"] = _codes(n, k, bits, group, "canonical", gen)
        state["out"] = torch.empty(n, k, dtype=_DTYPE[case["dtype"]], device="cuda")
        return state
    tiled = case["layout"] == "tiled"
    state["packed"], state["scales"] = _codes(n, k, bits, group, case["layout"], gen)
    state["b_layout"] = B.TILED if tiled else B.CANONICAL
    m = case.get("m", 1)
    x = _activations(m, k, case["dtype"], gen)
    if op == "gemv":
        state["x"], state["y"] = x[0], torch.empty(n, dtype=x.dtype, device="cuda")
        need = B.pot_gemv_workspace_bytes(n, k, bits, group) if tiled else 0
    else:
        state["x"], state["y"] = x, torch.empty(m, n, dtype=x.dtype, device="cuda")
        need = B.pot_gemm_workspace_bytes(m, n, k, bits, group) if tiled else 0
    state["ws"] = B.new_workspace(need)
    return state


def run(state: dict):
    s, op = state, state["op"]
    if op == "decode":
        s["graph"].replay()
        return s["ys"]
    if op == "gemv":
        return B.pot_gemv(s["packed"], s["scales"], s["k"], s["bits"], s["group"], s["x"], s["b_layout"], y=s["y"], workspace=s["ws"])
    if op == "gemm":
        return B.pot_gemm(s["packed"], s["scales"], s["k"], s["bits"], s["group"], s["x"], s["b_layout"], Y=s["y"], workspace=s["ws"])
    if op == "dequant":
        return B.pot_dequant(s["packed"], s["scales"], s["k"], s["bits"], s["group"], B.F16 if s["dtype"] == "f16" else B.BF16, out=s["out"])
    packed, scales = B.pot_quantize_ref(s["w"], s["bits"], s["group"], _RULE[s["rule"]])
    return packed, scales, B.pot_repack(packed, s["k"], s["bits"], 0), B.pot_repack_scales(scales, s["k"], s["group"], 0)


def _code_bytes(n: int, k: int, bits: int, group: int) -> int:
    return n * k * bits // 8 + n * (k // group) * 2


def work(case: dict) -> dict:
    op, bits, group = case["op"], case["bits"], case["group"]
    if op == "decode":
        h, f = case["hidden"], case["ffn"]
        shapes = ((3 * h, h), (h, h), (f, h), (f, h), (h, f))
        return dict(bytes=case["layers"] * sum(_code_bytes(n, k, bits, group) + 2 * n + 2 * k for n, k in shapes),
                    flops=case["layers"] * sum(2 * n * k for n, k in shapes))
    n, k = case["n"], case["k"]
    codes = _code_bytes(n, k, bits, group)
    if op == "encode":  # FP16 weights in; canonical and tiled codes and scales out
        return dict(bytes=2 * n * k + 2 * codes, flops=0)
    if op == "dequant":
        return dict(bytes=codes + 2 * n * k, flops=0)
    m = case.get("m", 1)
    return dict(bytes=codes + 2 * m * (n + k), flops=2 * m * n * k)


def tolerance(case: dict):
    """Codes, scales and unpacked weights are bit-exact.  Products: sums in FP32 (exact products), one rounding to the
    activations' type at the end; against the same sums in FP64 before that rounding the relative error is that of the
    rounding, 2^-11 / sqrt(3) * 0.7 for FP16 and eight times as much for BF16 (measured 2.1e-4 and 1.7e-3); four times that."""
    if case["op"] in ("encode", "dequant"):
        return "exact"
    return {"rel": 7e-3} if case.get("dtype") == "bf16" else {"rel": 8e-4}


def _pot_values(n: int, k: int, bits: int, group: int, dtype: str, gen: torch.Generator) -> torch.Tensor:
    """The weights that `_codes` stands for, [n, k] FP64, from the format's definition: sign * 2^E * scale with the top level on
    the group's largest magnitude, the scale an FP16 number (rounded once to BF16 for BF16 products)."""
    w, qmax = _weights(n, k, gen), (1 << (bits - 1)) - 1
    out = torch.empty(n, k, dtype=torch.float64, device="cuda")
    for r in range(0, n, 2048):
        g = w[r:r + 2048].double().view(-1, k // group, group)
        s = (g.abs().amax(2, keepdim=True) * 2.0 ** -qmax).clamp(2.0 ** -14, (2 - 2.0 ** -10) * 2.0 ** (15 - qmax)).to(torch.float16).double()
        level = torch.ones_like(g)
        for e in range(qmax):  # |w| / s above 2^(e + 1/2)
            level = torch.where(g * g > s * s * 2.0 ** (2 * e + 1), 2.0 ** (e + 1), level)
        if dtype == "bf16":
            s = s.to(torch.bfloat16).double()
        out[r:r + 2048] = torch.where(g < 0, -level, level).mul_(s).view(-1, k)
    return out


def exact(case: dict, seed: int):
    """What `run` returns for these inputs, in FP64 from plain torch; the encoder's results are whole numbers."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    op, bits, group = case["op"], case["bits"], case["group"]
    if op == "encode":
        return None
    if op == "decode":
        h, f = case["hidden"], case["ffn"]
        ys = []
        for _ in range(case["layers"]):
            for n, k in ((3 * h, h), (h, h), (f, h), (f, h), (h, f)):
                w = _pot_values(n, k, bits, group, "f16", gen)
                ys.append(w @ _activations(1, k, "f16", gen)[0].double())
        return ys
    w = _pot_values(case["n"], case["k"], bits, group, case["dtype"], gen)
    if op == "dequant":
        return w
    x = _activations(case.get("m", 1), case["k"], case["dtype"], gen).double()
    return w @ x[0] if op == "gemv" else x @ w.T
