"""The work a user of this library has it do, as cases that can be timed and compared between two builds.

A case is a dict of plain values:
  op      which entry points a pass goes through (below)
  M       activation rows (tokens)
  shapes  "NxK" of each weight tensor of the pass, comma separated; the pass takes them in order
  layers  how many times that list is repeated with weights of its own (1 where absent)
  block   elements per weight scale block (16 where absent)
  aware   scale-aware special-value selection in the weight quantizer (False where absent)

Operations:
  gemv        razer_gemv, one call per weight tensor, launched from the host
  gemv_graph  the same calls captured once into a CUDA graph and replayed, which is how a decode loop is served
  gemv_host   razer_gemv_host: activations come from pinned host memory and the result goes back there
  gemm        razer_gemm (prefill)
  w4a4        razer_quant_act, then razer_gemm_w4a4 (both operands RaZeR, exact bf16 route)
  w4a4_native razer_quant_act without a special value, then razer_gemm_w4a4 on the block-scaled FP4 instruction
  w4a4_fp4    razer_quant_act_fp4, then razer_gemm_w4a4_fp4 (the quantizer writes the operand the matmul reads)
  quantize    razer_quant_weight, razer_pack_layout and razer_dequant: a weight tensor is quantized, laid out for the
              kernels, and decoded to bf16 as accuracy studies with dequantized weights need it

Weights are Student-t (nu = 5) x 0.02 with 0.1 % of the entries ten times larger, quantized by the library; activations
are N(0, 1) in bf16 with 1 % of the channels twenty times larger.  Buffers and workspaces are allocated once, as a
serving loop keeps them.
"""
import math

import torch

from paper_2501_04052_b200 import binding as b

LLAMA7B = "4096x4096,11008x4096,4096x11008"


def listed():
    return [
        # One small layer, one token: what a call costs when there is next to nothing to compute.
        {"name": "gemv_small", "op": "gemv", "M": 1, "shapes": "1024x1024"},
        # One decode step of four Llama-7B-shaped layers for one sequence; 136 MB of weights, so they come from HBM.
        {"name": "decode_step", "op": "gemv_graph", "M": 1, "shapes": LLAMA7B, "layers": 4},
        # The same for a caller whose activations live on the host (a pipeline stage, an offloading runtime).
        {"name": "decode_host", "op": "gemv_host", "M": 1, "shapes": "4096x11008"},
        # Decode of a few sequences at once against the largest 70B-like projections.
        {"name": "decode_m4", "op": "gemv", "M": 4, "shapes": "28672x8192"},
        {"name": "decode_m16", "op": "gemv", "M": 16, "shapes": "8192x28672"},
        # A full decode batch against an attention-sized projection.
        {"name": "decode_m64", "op": "gemv", "M": 64, "shapes": "8192x8192"},
        # Ragged in every dimension: rows and columns that fill no tile, an odd batch (vocabulary slices, pruned layers).
        {"name": "decode_ragged", "op": "gemv", "M": 7, "shapes": "3333x2064"},
        # Prefill of a full prompt, and of a short odd-sized one.
        {"name": "prefill", "op": "gemm", "M": 2048, "shapes": "14336x4096"},
        {"name": "prefill_ragged", "op": "gemm", "M": 333, "shapes": "4096x11008"},
        # Weight-activation path: quantize the activations on the fly, multiply; the exact route at a mixed batch, the
        # FP4 tensor-core route on a prompt.
        {"name": "w4a4", "op": "w4a4", "M": 256, "shapes": "8192x8192"},
        {"name": "w4a4_fp4", "op": "w4a4_fp4", "M": 2048, "shapes": "8192x8192"},
        # Offline quantization of one MLP projection.
        {"name": "quantize", "op": "quantize", "M": 0, "shapes": "11008x4096"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: M, N and K spread over their logarithms, K a multiple of 16 (the format's
    block), nothing aligned beyond that in half of the draws."""
    op = rng.choice(["gemv", "gemv", "gemv_graph", "gemv_host", "gemm", "gemm", "w4a4", "w4a4_native", "w4a4_fp4", "quantize"])
    aligned = rng.random() < 0.5
    while True:
        n, k = _log_int(rng, 256, 28672), _log_int(rng, 256, 28672)
        if aligned:
            n, k = max(256, n // 256 * 256), max(256, k // 256 * 256)
        else:
            k = max(256, k // 16 * 16)
        if n * k <= 28672 * 8192:
            break
    c = {"op": op, "shapes": "%dx%d" % (n, k)}
    if op in ("gemv", "gemv_graph", "gemv_host"):
        c["M"] = 1 if rng.random() < 0.3 else _log_int(rng, 1, 64)
        if op == "gemv_graph":
            c["layers"] = max(1, min(4, (28672 * 8192) // (n * k)))
    elif op == "quantize":
        n = max(1, min(n, 11008 * 4096 // k))
        c["block"] = rng.choice([16, 16, 32, 64, 128])
        k = max(c["block"], k // c["block"] * c["block"])
        c["shapes"] = "%dx%d" % (n, k)
        c["M"] = 0
        c["aware"] = rng.random() < 0.25
    else:
        most = min(2048, 2048 * 14336 * 4096 // (n * k))
        c["M"] = _log_int(rng, min(65 if op == "gemm" else 16, most), most)
    return c


def _shapes(case):
    one = [tuple(int(v) for v in s.split("x")) for s in case["shapes"].split(",")]
    return one * int(case.get("layers", 1))


def _student_t(n, k, gen):
    z = torch.randn((n, k), generator=gen, device="cuda")
    chi = torch.zeros_like(z)
    for _ in range(5):
        chi.addcmul_(t := torch.randn((n, k), generator=gen, device="cuda"), t)
    w = z.mul_(0.02).div_(chi.div_(5.0).sqrt_())
    return torch.where(torch.rand((n, k), generator=gen, device="cuda") < 0.001, w * 10.0, w)


def _activations(m, k, gen):
    x = torch.randn((m, k), generator=gen, device="cuda")
    loud = torch.randperm(k, generator=gen, device="cuda")[: -(-k // 100)]
    x[:, loud] *= 20.0
    return x.to(torch.bfloat16)


def _weights(n, k, gen, block):
    codes, scales, ts = b.razer_quant_weight(_student_t(n, k, gen), block=block)
    desc = b.make_desc(n, k, float(ts.item()), block=block)
    return desc, b.razer_pack_layout(desc, codes, scales)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    op, m, block = case["op"], int(case["M"]), int(case.get("block", 16))
    state = {"op": op, "M": m, "block": block, "aware": bool(case.get("aware", False))}
    if op == "quantize":
        (n, k), = _shapes(case)
        state["w"] = _student_t(n, k, gen)
        return state
    code = {"gemm": b.OP_GEMM, "w4a4": b.OP_GEMM_W4A4, "w4a4_native": b.OP_GEMM_W4A4, "w4a4_fp4": b.OP_GEMM_W4A4}.get(op, b.OP_GEMV)
    calls = []
    for n, k in _shapes(case):
        desc, packed = _weights(n, k, gen, block)
        x = _activations(m, k, gen)
        y = torch.empty((m, n), dtype=torch.bfloat16, device="cuda")
        call = {"desc": desc, "packed": packed, "x": x, "y": y, "ws": b.alloc_workspace(desc, m, code, "cuda")}
        if op == "gemv_host":
            call["x_host"], call["y_host"] = x.cpu().pin_memory(), torch.empty((m, n), dtype=torch.bfloat16).pin_memory()
        if op == "w4a4_fp4":
            call["act"] = torch.empty(b.razer_fp4_act_bytes(m, k), dtype=torch.uint8, device="cuda")
        if op.startswith("w4a4"):
            call["scratch"] = torch.zeros(2, dtype=torch.int32, device="cuda")
        calls.append(call)
    state["calls"] = calls
    if op == "gemv_graph":
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _gemv(calls)
        torch.cuda.current_stream().wait_stream(side)
        state["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(state["graph"]):
            _gemv(calls)
    return state


def _gemv(calls):
    return [b.razer_gemv(c["desc"], c["packed"], c["x"], c["y"], c["ws"]) for c in calls]


def run(state):
    op = state["op"]
    if op == "quantize":
        codes, scales, ts = b.razer_quant_weight(state["w"], block=state["block"], scale_aware=state["aware"])
        n, k = state["w"].shape
        desc = b.make_desc(n, k, float(ts.item()), block=state["block"])
        packed = b.razer_pack_layout(desc, codes, scales)
        return codes, scales, ts, b.razer_dequant(desc, packed, fp32=False)
    calls = state["calls"]
    if op == "gemv":
        return _gemv(calls)
    if op == "gemv_graph":
        state["graph"].replay()
        return [c["y"] for c in calls]
    if op == "gemv_host":
        for c in calls:
            b.razer_gemv_host(c["desc"], c["packed"], c["x_host"], c["y_host"], c["x"], c["y"], c["ws"])
        return [c["y_host"] for c in calls]
    if op == "gemm":
        return [b.razer_gemm(c["desc"], c["packed"], c["x"], c["y"], c["ws"]) for c in calls]
    out = []
    for c in calls:
        if op == "w4a4_fp4":
            act, ts = b.razer_quant_act_fp4(c["x"], act_fp4=c["act"], scratch=c["scratch"])
            out.append((b.razer_gemm_w4a4_fp4(c["desc"], c["packed"], act, ts, state["M"], y=c["y"], workspace=c["ws"]), ts))
        else:
            native = op == "w4a4_native"
            codes, scales, ts = b.razer_quant_act(c["x"], sv_mag=0.0 if native else 5.0, scratch=c["scratch"])
            y = b.razer_gemm_w4a4(c["desc"], c["packed"], codes, scales, ts, y=c["y"], workspace=c["ws"], use_native_fp4=native)
            out.append((y, codes, scales, ts))
    return out


def work(case):
    m, total, flops = int(case["M"]), 0.0, 0.0
    for n, k in _shapes(case):
        weights = n * k * 0.5 + n * k / 16.0
        if case["op"] == "quantize":
            # FP32 in; codes, scale bytes and the bf16 tensor out
            total += 4.0 * n * k + n * k * 0.5 + n * k / int(case.get("block", 16)) + 2.0 * n * k
            continue
        total += weights + 2.0 * m * k + 2.0 * m * n
        if case["op"] in ("w4a4", "w4a4_native"):
            total += m * k * 0.5625
        flops += 2.0 * m * n * k
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """Quantized codes, scale bytes and decoded weights are exact.  A matmul output is an FP32 sum rounded to bf16 once:
    another order of the sum moves a few outputs across a rounding boundary by one bf16 unit (at most 2^-7 = 7.8e-3 of the
    value).  Measured against the same product in 64 bits: up to 1.8e-4 in the 2-norm, 7.8e-3 at the worst element."""
    if case["op"] == "quantize":
        return "exact"
    return {"rel": 7e-4, "max": 1e-2}
