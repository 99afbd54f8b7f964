"""What a user of this library has it do, as cases that can be prepared, run and compared.

The public entry points are those of ``paper_2601_16536_b200.binding``: the product C = A . Dequant(W) on
packed 4-bit weights with the activations on the device (``w4a16_gemm``) or on the host
(``w4a16_gemm_host``), the quantizer and the offline reorder that a model load goes through
(``w4a16_quantize``, ``w4a16_pack``), and the standalone dequantization (``w4a16_dequant``).

Case fields
  kind        "gemm", "host" (activations and result in pinned host memory), "quantize_pack" or "dequant"
  layers      weight matrices of one pass, "KxN" separated by commas; one call each
  M           batch rows (0 where there are none)
  group       quantization group along K: 32, 64 or 128
  symmetric   zero point fixed at 8, no zero points stored
  bf16        BF16 activations, scales, dequantized weights and results instead of FP16
  bias, act   optional step fused into the final rounding; act as in the C ABI (0 none, 1 ReLU, 2 SiLU)
  sigma, outliers   activations ~ N(0, sigma); with outliers 1 % of the K columns are twenty times larger
"""
import math

import torch

from paper_2601_16536_b200 import binding as B

# The linear layers of one transformer block: fused QKV, output projection, gate + up, down.
BLOCK = "4096x12288,4096x4096,4096x22016,11008x4096"

_workspace = None   # Split-K scratch: one per process, grown when a shape needs more, as a serving program keeps it


def _case(name, kind, layers, M, group=128, symmetric=False, bf16=False, bias=False, act=0, sigma=1.0, outliers=False):
    return {"name": name, "kind": kind, "layers": layers, "M": M, "group": group, "symmetric": symmetric, "bf16": bf16,
            "bias": bias, "act": act, "sigma": sigma, "outliers": outliers}


def listed():
    return [
        # one small layer for one token: nothing but the latency of a call
        _case("decode_one_layer_m1", "gemm", "4096x4096", 1),
        # one token through the linear layers of a transformer block: single-stream generation
        _case("decode_block_m1", "gemm", BLOCK, 1),
        # sixteen sequences generating together
        _case("decode_block_m16", "gemm", BLOCK, 16),
        # a down projection with K much larger than N, few sequences, outlier channels
        _case("decode_long_k_m4", "gemm", "28672x8192", 4, sigma=0.5, outliers=True),
        # the same layer under a larger batch
        _case("batch_long_k_m32", "gemm", "28672x8192", 32, sigma=0.5, outliers=True),
        # a busy server's decode batch, or a short prompt, through a block
        _case("batch_block_m64", "gemm", BLOCK, 64),
        # a short prompt on a layer with K four times N
        _case("prefill_long_k_m256", "gemm", "16384x4096", 256),
        # a prompt of odd length in the other formats: BF16, symmetric, groups of 64, bias and SiLU in the same call
        _case("prefill_bf16_sym_g64_silu_m777", "gemm", "4096x22016", 777, group=64, symmetric=True, bf16=True, bias=True, act=2),
        # a long prompt: compute-bound
        _case("prefill_m4096", "gemm", "8192x8192", 4096),
        # activations and result in host memory, copies and product in one call
        _case("host_buffers_m8", "host", "11008x4096", 8),
        # loading a layer: 16-bit weights to codes, scales and zero points, and those to the kernels' layout
        _case("load_quantize_pack", "quantize_pack", "11008x4096", 0),
        # the weights back in 16 bits: checks, fine-tuning, layers that are not run quantized
        _case("dequantize", "dequant", "8192x8192", 0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """K a multiple of 128 from 1024 to 28672, N a multiple of 64 (odd multiples too) from 1024 to 28672, M from
    1 to 4096 (up to 16 from host memory), every format; never more weights or more arithmetic than the largest
    listed cases."""
    kind = rng.choice(["gemm"] * 7 + ["host", "quantize_pack", "dequant"])
    while True:
        K = 128 * _log_int(rng, 8, 224)
        N = 64 * _log_int(rng, 16, 448)
        M = {"gemm": _log_int(rng, 1, 4096), "host": _log_int(rng, 1, 16)}.get(kind, 0)
        if K * N <= (28672 * 8192 if kind in ("gemm", "host") else 8192 * 8192) and M * K * N <= 4096 * 8192 * 8192:
            break
    plain = kind == "host"      # (the host form takes the benchmark's format only)
    c = _case("", kind, "%dx%d" % (K, N), M, group=rng.choice([32, 64, 128]) if not plain else 128,
              symmetric=not plain and rng.random() < 0.3, bf16=not plain and rng.random() < 0.3)
    if kind == "gemm":
        c["bias"] = rng.random() < 0.25
        c["act"] = rng.choice([0, 0, 0, 1, 2])
        c["sigma"] = rng.choice([0.5, 1.0])
        c["outliers"] = rng.random() < 0.25
    del c["name"]
    return c


def _shapes(case):
    return [tuple(int(x) for x in s.split("x")) for s in case["layers"].split(",")]


def _flags(case):
    return (B.FLAG_SYMMETRIC if case["symmetric"] else 0) | (B.FLAG_BF16 if case["bf16"] else 0)


def _dtype(case):
    return torch.bfloat16 if case["bf16"] else torch.float16


def _packed(case, K, N, gen):
    """A packed weight matrix with uniform codes and zero points and scales ~ U[0.002, 0.02]."""
    g = case["group"]
    Wq = torch.randint(-2 ** 31, 2 ** 31, (K // 8, N), generator=gen, device="cuda", dtype=torch.int32)
    S = torch.empty((K // g, N), device="cuda").uniform_(0.002, 0.02, generator=gen).to(_dtype(case))
    Z = None
    if not case["symmetric"]:
        Z = torch.randint(0, 16, (K // g, N), generator=gen, device="cuda", dtype=torch.uint8)
    return B.w4a16_pack(Wq, S, Z, N, K, g, _flags(case))


def _activations(case, K, gen):
    A = torch.randn((case["M"], K), generator=gen, device="cuda") * case["sigma"]
    if case["outliers"]:
        A[:, torch.randperm(K, generator=gen, device="cuda")[: round(0.01 * K)]] *= 20.0
    return A.to(_dtype(case))


def _reserve_workspace(nbytes):
    global _workspace
    if _workspace is None or _workspace.numel() < nbytes:
        torch.cuda.synchronize()
        _workspace = B.ensure_workspace(nbytes)


def prepare(case, seed):
    """Inputs from the seed, packed weights, and the output buffers that such a program keeps."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    kind, M, state = case["kind"], case["M"], {"case": case, "calls": []}
    for K, N in _shapes(case):
        if kind == "quantize_pack":
            W = torch.randn((K, N), generator=gen, device="cuda") * 0.04
            W[::97, ::5] *= 6.0                                   # a few outliers per group
            state["calls"].append({"W": W.to(_dtype(case))})
            continue
        call = {"pw": _packed(case, K, N, gen)}
        if kind == "dequant":
            call["out"] = torch.empty((K, N), dtype=_dtype(case), device="cuda")
        else:
            _reserve_workspace(B.w4a16_workspace_bytes(M, N, K, case["group"], 0))
            call["A"] = _activations(case, K, gen)
            call["C"] = torch.empty((M, N), dtype=_dtype(case), device="cuda")
            call["bias"] = torch.randn(N, generator=gen, device="cuda").to(_dtype(case)) if case["bias"] else None
        if kind == "host":
            call["A_host"] = call["A"].cpu().pin_memory()
            call["A"].zero_()                                      # the staging buffer of the call
            call["C_host"] = torch.zeros((M, N), dtype=_dtype(case)).pin_memory()
        state["calls"].append(call)
    return state


def run(state):
    case, out = state["case"], []
    for c in state["calls"]:
        if case["kind"] == "gemm":
            out.append(B.w4a16_gemm(c["A"], c["pw"], C=c["C"], bias=c["bias"], act=case["act"]))
        elif case["kind"] == "host":
            B.w4a16_gemm_host(c["A_host"], c["A"], c["pw"], c["C"], c["C_host"])
            out.append(c["C_host"])
        elif case["kind"] == "quantize_pack":
            Wq, S, Z = B.w4a16_quantize(c["W"], case["group"], _flags(case))
            K, N = c["W"].shape
            pw = B.w4a16_pack(Wq, S, Z, N, K, case["group"], _flags(case))
            out.append((Wq, S, Z, pw.Wq, pw.S, pw.Z))
        else:
            out.append(B.w4a16_dequant(c["pw"], out=c["out"]))
    return out


def work(case):
    M, g = case["M"], case["group"]
    nbytes = flops = 0
    for K, N in _shapes(case):
        scales, zeros = 2 * (K // g) * N, 0 if case["symmetric"] else (K // g) * N
        packed = K * N // 2 + scales + zeros // 2
        if case["kind"] == "quantize_pack":     # 16-bit weights in; codes, scales, zero points and the packed form out
            nbytes += 2 * K * N + K * N // 2 + scales + zeros + packed
        elif case["kind"] == "dequant":
            nbytes += packed + 2 * K * N
        else:
            nbytes += packed + 2 * M * (K + N) + (2 * N if case["bias"] else 0)
            flops += 2 * M * N * K
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    # Codes, zero points, packed words and dequantized weights are decided bit by bit.
    if case["kind"] in ("quantize_pack", "dequant"):
        return "exact"
    # A product: the weights are rounded to 16 bits by definition, the sums are FP32, the result is rounded once
    # to 16 bits.  Against the same product in 64 bits (dequantized weights, listed cases and 40 drawn ones) the
    # path shows rel 2.02e-4 to 2.1e-4 and max 4.7e-4 to 5.2e-4 in FP16, rel 1.65e-3 to 1.68e-3 and max 3.6e-3 to
    # 3.9e-3 in BF16, all of it the last rounding: four times that.
    return {"rel": 6.6e-3, "max": 1.6e-2} if case["bf16"] else {"rel": 8.3e-4, "max": 2.0e-3}
