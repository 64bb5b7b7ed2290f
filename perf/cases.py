"""The work that a user of this library has it do, as timed cases: decode steps, prompts, the integer path of
ternary weights, and packing a checkpoint, each through the entry points of `paper_2511_11248_b200.binding`.

A case is a dict of plain values:
  op      "decode"          decode calls of one or more decoder layers, M in 1..8 (tman_mpgemv, tman_mpgemv_grouped)
          "prefill"         one prompt through one projection (tman_mpgemm)
          "ternary_decode"  row quantization + integer decode of the up and down projection (tman_quantize_rows,
                            tman_mpgemv_ternary)
          "ternary_prefill" row quantization + INT8 prefill of one projection (tman_quantize_rows_i8,
                            tman_mpgemm_ternary_i8)
          "pack"            one weight matrix into the packed layout (tman_pack_weights)
  M, bits, group, and K, N (one matrix) or hidden, kv, ffn, layers (decoder layers; "part" says which projections)
  graph   the calls are captured once in a CUDA graph and a pass replays it, as a program that generates
          token after token does (the decode default of bench.py); otherwise they are issued one by one
Weights and activations are synthetic with the distributions of `synth.py`, drawn on the device.
"""
import math

import torch

from paper_2511_11248_b200 import binding as B

MAX_FLOPS = 2.0 * 8192 * 3584 * 18944      # the largest listed case
BITNET = (2560, 6912)                      # hidden and inner size of the ternary model shapes
W_SCALE = 0.0173


def listed():
    return [
        # One small projection (key or value of a 4096-wide layer), one token, issued eagerly: the smallest call
        # there is; launch cost and fixed phases.
        dict(name="decode_kv_proj_m1", op="decode", part="single", graph=False, M=1, K=4096, N=1024, bits=4, group=64, layers=1),
        # The benchmark's default workload: the 2-bit MLP (gate and up in one grouped call, down), one token; four
        # layers of it, so that weights stream from HBM as they do in a model.
        dict(name="decode_mlp_m1_b2", op="decode", part="mlp", graph=True, M=1, hidden=4096, kv=1024, ffn=14336, bits=2, group=64, layers=4),
        # Whole decoder layers, one token: the chat case of single-user generation with 4-bit weights.
        dict(name="decode_layer_m1_b4", op="decode", part="layer", graph=True, M=1, hidden=4096, kv=1024, ffn=14336, bits=4, group=128, layers=2),
        # A few sequences (or a short speculative draft) at once, 3-bit.
        dict(name="decode_layer_m4_b3", op="decode", part="layer", graph=True, M=4, hidden=4096, kv=1024, ffn=14336, bits=3, group=64, layers=2),
        # The widest decode batch the decode call takes, 4-bit.
        dict(name="decode_layer_m8_b4", op="decode", part="layer", graph=True, M=8, hidden=4096, kv=1024, ffn=14336, bits=4, group=128, layers=2),
        # A batch just beyond the decode call's eight rows, or a very short prompt, ragged.
        dict(name="prefill_m40_b4", op="prefill", graph=False, M=40, K=4096, N=14336, bits=4, group=128),
        # A 128-token prompt (the sequence length the paper's GEMM kernels are quoted at).
        dict(name="prefill_m128_b4", op="prefill", graph=False, M=128, K=3584, N=18944, bits=4, group=128),
        # An ordinary prompt of odd length through an attention projection, 2-bit.
        dict(name="prefill_m777_b2", op="prefill", graph=False, M=777, K=3584, N=4608, bits=2, group=64),
        # A long batch of prompts through the longest reduction.
        dict(name="prefill_m8192_b4", op="prefill", graph=False, M=8192, K=18944, N=3584, bits=4, group=128),
        # Ternary (BitNet-like) MLP, one token: 16-bit integer activations.
        dict(name="ternary_decode_m1", op="ternary_decode", graph=True, M=1, K=2560, N=6912, bits=2, group=128, layers=4),
        # The same model's prompt: INT8 activations.
        dict(name="ternary_prefill_m2048", op="ternary_prefill", graph=False, M=2048, K=2560, N=6912, bits=2, group=128),
        # Loading a model: one large matrix repacked.
        dict(name="pack_b4", op="pack", graph=False, M=1, K=4096, N=14336, bits=4, group=128),
    ]


def _log(rng, lo, hi, step):
    """A multiple of `step` in [lo, hi], spread over the logarithm."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return int(min(hi // step * step, max(-(-lo // step) * step, round(v / step) * step)))


def draw(rng):
    op = rng.choice(["decode", "decode", "decode", "prefill", "prefill", "prefill", "ternary_decode", "ternary_prefill", "pack"])
    bits, group = rng.choice([2, 3, 4]), rng.choice([32, 64, 128, 64, 128])
    if op == "decode":
        M = rng.randint(1, 8)
        part = rng.choice(["single", "mlp", "layer", "layer"])
        if part == "single":
            return dict(op=op, part=part, graph=rng.random() < 0.5, M=M, K=_log(rng, 1024, 18944, 128), N=_log(rng, 256, 18944, 8),
                        bits=bits, group=group, layers=1)
        hidden = _log(rng, 1536, 5120, 128)
        return dict(op=op, part=part, graph=True, M=M, hidden=hidden, kv=_log(rng, hidden // 8, hidden, 8),
                    ffn=_log(rng, 2 * hidden, 4 * hidden, 128), bits=bits, group=group, layers=rng.randint(1, 4))
    if op in ("ternary_decode", "ternary_prefill"):
        K, N = _log(rng, 1536, 6912, 128), _log(rng, 1536, 8192, 128)
        if op == "ternary_decode":
            return dict(op=op, graph=True, M=rng.randint(1, 8), K=K, N=N, bits=2, group=group, layers=rng.randint(1, 4))
        return dict(op=op, graph=False, M=_log(rng, 64, 4096, 1), K=K, N=N, bits=2, group=group)
    K, N = _log(rng, 1024, 18944, 128), _log(rng, 512, 18944, 8)
    if op == "pack":
        return dict(op=op, graph=False, M=1, K=K, N=N, bits=bits, group=group)
    return dict(op=op, graph=False, M=min(_log(rng, 9, 8192, 1), int(MAX_FLOPS / (2.0 * K * N))), K=K, N=N, bits=bits, group=group)


def _calls(case):
    """The decode calls of one layer: (K, output widths of the matrices that share the activations)."""
    if case["op"] == "ternary_decode":
        return [(case["K"], [case["N"]]), (case["N"], [case["K"]])]
    if case.get("part", "single") == "single":
        return [(case["K"], [case["N"]])]
    h, kv, f = case["hidden"], case["kv"], case["ffn"]
    mlp = [(h, [f, f]), (f, [h])]
    return mlp if case["part"] == "mlp" else [(h, [h, kv, kv]), (h, [h])] + mlp


def _weights(gen, K, N, bits, group):
    codes = torch.randint(0, 1 << bits, (K, N), dtype=torch.uint8, device="cuda", generator=gen)
    zeros = torch.randint(0, 1 << bits, (K // group, N), dtype=torch.uint8, device="cuda", generator=gen)
    lo, hi = (0.01, 0.05) if bits == 2 else (0.005, 0.02)
    scales = (lo + (hi - lo) * torch.rand((K // group, N), device="cuda", generator=gen)).to(torch.float16)
    return codes, scales, zeros


def _packed(gen, K, N, bits, group):
    codes, scales, zeros = _weights(gen, K, N, bits, group)
    packed = torch.empty(B.tman_packed_bytes(K, N, bits, group), dtype=torch.uint8, device="cuda")
    B.tman_pack_weights(codes, scales, zeros, K, N, bits, group, packed)
    return packed


def _packed_ternary(gen, K, N, group):
    # thirds of -1, 0, +1 as codes 0, 1, 2; the buffer's scales and zero-points are implied by the path
    codes = torch.randint(0, 3, (K, N), dtype=torch.uint8, device="cuda", generator=gen)
    packed = torch.empty(B.tman_packed_bytes(K, N, 2, group), dtype=torch.uint8, device="cuda")
    B.tman_pack_weights(codes, torch.ones((K // group, N), dtype=torch.float16, device="cuda"),
                        torch.ones((K // group, N), dtype=torch.uint8, device="cuda"), K, N, 2, group, packed)
    return packed


def _workspace(nbytes):
    ws = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    B.tman_workspace_init(ws)
    return ws


def _half(*shape):
    return torch.empty(shape, dtype=torch.float16, device="cuda")


def _activations(gen, M, K, outliers=False):
    x = torch.randn((M, K), device="cuda", generator=gen)
    if outliers:                                   # a seeded 1 % of the channels twenty times as large
        x[:, torch.randperm(K, device="cuda", generator=gen)[:max(1, K // 100)]] *= 20.0
    return x.to(torch.float16)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    op, M, bits, group = case["op"], case["M"], case["bits"], case["group"]
    st = {"case": case, "graph": None}
    if op in ("decode", "ternary_decode"):
        calls = _calls(case)
        if op == "decode":
            ws = _workspace(max(B.tman_workspace_bytes(B.OP_GEMV, M, K, sum(Ns), bits, group) for K, Ns in calls))
        else:
            ws = _workspace(max(B.tman_workspace_bytes(B.OP_TERNARY, M, K, Ns[0], bits, group) for K, Ns in calls))
        st["ws"], st["steps"] = ws, []
        for _ in range(case["layers"]):
            for K, Ns in calls:
                step = {"K": K, "Ns": Ns, "x": _activations(gen, M, K), "y": [_half(M, N) for N in Ns]}
                if op == "decode":
                    step["packed"] = [_packed(gen, K, N, bits, group) for N in Ns]
                else:
                    step["packed"] = [_packed_ternary(gen, K, Ns[0], group)]
                    step["a"] = torch.empty((M, K), dtype=torch.int16, device="cuda")
                    step["s"] = torch.empty(M, dtype=torch.float32, device="cuda")
                st["steps"].append(step)
        if case["graph"]:
            _issue_decode(st)                      # a first pass outside the capture, as a program warms up
            torch.cuda.synchronize()
            st["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(st["graph"]):
                _issue_decode(st)
        return st
    K, N = case["K"], case["N"]
    if op == "pack":
        st["in"] = _weights(gen, K, N, bits, group)
        st["packed"] = torch.empty(B.tman_packed_bytes(K, N, bits, group), dtype=torch.uint8, device="cuda")
        return st
    st["x"], st["y"] = _activations(gen, M, K, outliers=True), _half(M, N)
    if op == "prefill":
        st["packed"] = _packed(gen, K, N, bits, group)
        st["ws"] = _workspace(B.tman_workspace_bytes(B.OP_GEMM, M, K, N, bits, group))
    else:
        st["packed"] = _packed_ternary(gen, K, N, group)
        st["ws"] = _workspace(B.tman_workspace_bytes(B.OP_AUX, M, K, N, bits, group))
        st["a"] = torch.empty((M, K), dtype=torch.int8, device="cuda")
        st["s"] = torch.empty(M, dtype=torch.float32, device="cuda")
    return st


def _issue_decode(st):
    c, ws = st["case"], st["ws"]
    M, bits, group = c["M"], c["bits"], c["group"]
    for s in st["steps"]:
        if c["op"] == "ternary_decode":
            B.tman_quantize_rows(s["x"], M, s["K"], 32767, s["a"], s["s"])
            B.tman_mpgemv_ternary(s["packed"][0], s["a"], s["s"], W_SCALE, s["y"][0], None, M, s["K"], s["Ns"][0], group, ws)
        elif len(s["Ns"]) == 1:
            B.tman_mpgemv(s["packed"][0], s["x"], s["y"][0], M, s["K"], s["Ns"][0], bits, group, ws)
        else:
            B.tman_mpgemv_grouped(s["packed"], s["x"], s["y"], M, s["K"], s["Ns"], bits, group, ws)


def run(state):
    c = state["case"]
    op, M, bits, group = c["op"], c["M"], c["bits"], c["group"]
    if op in ("decode", "ternary_decode"):
        if state["graph"] is not None:
            state["graph"].replay()
        else:
            _issue_decode(state)
        return [y for s in state["steps"] for y in s["y"]]
    K, N = c["K"], c["N"]
    if op == "pack":
        codes, scales, zeros = state["in"]
        B.tman_pack_weights(codes, scales, zeros, K, N, bits, group, state["packed"])
        return state["packed"]
    if op == "prefill":
        B.tman_mpgemm(state["packed"], state["x"], state["y"], M, K, N, bits, group, state["ws"])
    else:
        B.tman_quantize_rows_i8(state["x"], M, K, state["a"], state["s"])
        B.tman_mpgemm_ternary_i8(state["packed"], state["a"], state["s"], W_SCALE, state["y"], M, K, N, group, state["ws"])
    return state["y"]


def _matrix_bytes(K, N, bits, group):
    """Planes, scales and b-bit zero-points of one matrix."""
    return K * N * bits / 8 + (K // group) * N * (2 + bits / 8)


def work(case):
    op, M, bits, group = case["op"], case["M"], case["bits"], case["group"]
    if op in ("decode", "ternary_decode"):
        nbytes = flops = 0.0
        for K, Ns in _calls(case):
            nbytes += 2 * M * K
            for N in Ns:
                nbytes += 2 * M * N + (K * N / 4 if op == "ternary_decode" else _matrix_bytes(K, N, bits, group))
                flops += 2.0 * M * K * N
        return {"bytes": nbytes * case["layers"], "flops": flops * case["layers"]}
    K, N = case["K"], case["N"]
    if op == "pack":
        return {"bytes": K * N + (K // group) * N * 3 + _matrix_bytes(K, N, bits, group), "flops": 0.0}
    weights = _matrix_bytes(K, N, bits, group) if op == "prefill" else K * N / 4
    return {"bytes": weights + 2.0 * M * (K + N), "flops": 2.0 * M * K * N}


def tolerance(case):
    # About four times what the largest of 32 cases over the ranges above showed against the same product in 64 bits.
    op, M = case["op"], case["M"]
    if op == "pack":
        return "exact"
    if op in ("ternary_decode", "ternary_prefill"):
        # exact integer sums, two products in fp32 and one rounding to fp16
        return {"rel": 5e-4, "max": 2e-3}
    if op == "prefill":
        # weights rounded to fp16 once, fp32 sums, fp16 result: 2.9e-4 and 1.8e-3
        return {"rel": 1.2e-3, "max": 7e-3}
    if M == 1:
        # fp32 throughout, fp16 result: 2.3e-4 and 4.9e-4
        return {"rel": 9e-4, "max": 2e-3}
    # several rows may use fp16 table entries and fp16 sums inside 32 activations: 7.7e-4 and 3.5e-3
    return {"rel": 3e-3, "max": 1.4e-2}
