"""The work that users of the library have it do, as cases that can be timed through its public entry points.

A case names an entry point (`op`), a model and the sizes:

  dot       mmasim.dot_batch: n independent dot products, the shape of probe vectors
  gemm      mmasim.gemm: one whole matrix product under a model, on device tensors
  accuracy  accuracy.deviation_stats: a model's deviation from the FP64 result (model GEMM, reference GEMM, reduction)
  host      mmasim.gemm_host: a matrix product on pinned host buffers, copies in and out included

Results are words, so they have to be the same bit for bit; only the statistics of `accuracy`, whose sums run in no fixed
order, have a tolerance.
"""
import math

import torch

from paper_2511_10909_b200 import accuracy, mmasim

# One row per kind of arithmetic in the library: architecture, input type, accumulator type, elements per block of K.
GEMM_MODELS = [
    ("volta", "fp16", "fp32", 4), ("ampere", "fp16", "fp32", 8), ("hopper", "fp16", "fp32", 16), ("hopper", "fp16", "fp16", 16),
    ("ampere", "bf16", "fp32", 8), ("hopper", "bf16", "fp32", 16), ("ampere", "tf32", "fp32", 4), ("hopper", "tf32", "fp32", 8),
    ("ada", "e5m2", "fp32", 16), ("hopper", "e4m3", "fp32", 32), ("hopper", "e4m3", "fp16", 32), ("blackwell", "e4m3", "fp32", 32),
    ("blackwell", "e2m1", "fp32", 32), ("blackwell", "mxe4m3", "fp32", 32), ("blackwell", "mxf4", "fp32", 64),
    ("blackwell", "nvf4", "fp32", 64), ("cdna3", "bf16", "fp32", 8), ("cdna3", "tf32", "fp32", 4), ("cdna3", "e4m3", "fp32", 16),
    ("cdna1", "fp16", "fp32", 4), ("cdna1", "bf16", "fp32", 2), ("cdna2", "fp16", "fp32", 4), ("cdna2", "bf16", "fp32", 4),
    ("cdna1", "fp32", "fp32", 1), ("hopper", "fp64", "fp64", 1)]
DOT_MODELS = [("volta", "fp16", "fp32"), ("ampere", "fp16", "fp32"), ("hopper", "fp16", "fp32"), ("ampere", "bf16", "fp32"),
              ("hopper", "tf32", "fp32"), ("cdna2", "fp16", "fp32"), ("cdna2", "bf16", "fp32"), ("hopper", "e4m3", "fp32"),
              ("cdna3", "fp16", "fp32")]
ACCURACY_MODELS = [("hopper", "fp16", "fp32", 16), ("hopper", "e4m3", "fp32", 32), ("ampere", "bf16", "fp32", 8),
                   ("cdna3", "fp16", "fp32", 8), ("cdna2", "fp16", "fp32", 4)]
HOST_MODELS = [("hopper", "e4m3", "fp32", 32), ("hopper", "fp16", "fp32", 16), ("ampere", "bf16", "fp32", 8)]

BITS = {"fp64": 64, "fp32": 32, "tf32": 32, "bf16": 16, "fp16": 16, "mxf4": 4, "nvf4": 4}     # everything else: one byte
ACC_BYTES = {"fp64": 8, "fp32": 4, "fp16": 2}
WORDS = {8: torch.uint8, 16: torch.int16, 32: torch.int32, 64: torch.int64}
SCALE_BLOCK = {"mxe4m3": 32, "mxe5m2": 32, "mxf4": 32, "nvf4": 16}


def _case(op, model, M, N, K, **kw):
    return dict(op=op, arch=model[0], fmt=model[1], acc=model[2], M=M, N=N, K=K, **kw)


def listed():
    return [
        # a handful of probe vectors: the interactive call of someone working out what a unit does; nothing but latency
        dict(_case("dot", ("ampere", "fp16", "fp32"), 2048, 1, 16), name="dot_probe_small"),
        # the probe batch of the benchmark: 2^20 dots of length 32 with subnormals, cancellation, outliers, inf and NaN
        dict(_case("dot", ("hopper", "fp16", "fp32"), 1 << 20, 1, 32), name="dot_probe_batch"),
        # the smallest of the benchmark's matrix products: 256^3 with C = 0
        dict(_case("gemm", ("volta", "fp16", "fp32"), 256, 256, 256, c=False), name="gemm_volta_fp16_256"),
        # operand exponents spread over +-20 binades, so that alignment truncates most terms
        dict(_case("gemm", ("ampere", "bf16", "fp32"), 2048, 2048, 2048, c=True, dist="exponents"), name="gemm_ampere_bf16_2048"),
        # the benchmark's main workload
        dict(_case("gemm", ("hopper", "e4m3", "fp32"), 4096, 4096, 4096, c=True), name="gemm_hopper_e4m3_4096"),
        # the same unit with partial sums promoted to FP32 every 128 elements and per-row dequantisation scales
        dict(_case("gemm", ("hopper", "e4m3", "fp32"), 2048, 2048, 4096, c=False, k_chunk=128, scales=True), name="gemm_hopper_e4m3_promoted"),
        # a layer of a network while it generates: few rows, a whole weight matrix
        dict(_case("gemm", ("hopper", "fp16", "fp32"), 16, 4096, 4096, c=False), name="gemm_hopper_fp16_decode"),
        # sizes that nobody chose with tiles in mind
        dict(_case("gemm", ("ampere", "fp16", "fp32"), 1000, 1111, 1000, c=True), name="gemm_ampere_fp16_ragged"),
        # a layer of a network over a prompt, block-scaled FP8
        dict(_case("gemm", ("blackwell", "mxe4m3", "fp32"), 1024, 4096, 4096, c=False), name="gemm_blackwell_mxfp8_prefill"),
        # group-scaled FP4
        dict(_case("gemm", ("blackwell", "nvf4", "fp32"), 2048, 2048, 4096, c=False), name="gemm_blackwell_nvfp4"),
        # the analysis of a unit's bias: model, FP64 reference and the reduction of the deviations
        dict(_case("accuracy", ("cdna3", "fp16", "fp32"), 1024, 1024, 256, c=True), name="accuracy_cdna3_fp16"),
        # a caller whose matrices are in (pinned) host memory
        dict(_case("host", ("hopper", "e4m3", "fp32"), 2048, 2048, 2048, c=True), name="host_hopper_e4m3_2048"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _up(x, to):
    return -(-x // to) * to


def draw(rng):
    kind = rng.choices(["dot", "gemm", "accuracy", "host"], [4, 12, 2, 2])[0]
    if kind == "dot":
        return _case("dot", rng.choice(DOT_MODELS), _log(rng, 256, 1 << 20), 1, rng.choice([4, 8, 16, 32]))
    *model, block = rng.choice({"gemm": GEMM_MODELS, "accuracy": ACCURACY_MODELS, "host": HOST_MODELS}[kind])
    if kind == "gemm":
        M, N, K = (_log(rng, lo, 4096) for lo in (1, 16, 16))
    else:
        M, N, K = (_log(rng, 128, 2048) for _ in range(3))
    block = max(block, SCALE_BLOCK.get(model[1], 1))
    while M * N * K > 1 << 34:
        M, N, K = -(-M // 2), -(-N // 2), -(-K // 2)
    if rng.random() < 0.5:              # half of the sizes as networks have them, half as they come
        M, N, K = _up(M, 16) if M > 16 else M, _up(N, 64), _up(K, 128)
    else:
        K = _up(K, block)
    kw = {"c": rng.random() < 0.5}
    if kind == "gemm" and model[1] == "e4m3" and model[0] == "hopper" and model[2] == "fp32" and K % 128 == 0 and rng.random() < 0.5:
        kw.update(k_chunk=128, scales=True)
    return _case(kind, model, M, N, K, **kw)


# ---- inputs, made on the GPU ----
def _small_values(ebits, mbits, bias, codes, top):
    v = [(m / (1 << mbits)) * 2.0 ** (1 - bias) if e == 0 else (1 + m / (1 << mbits)) * 2.0 ** (e - bias)
         for e in range(1 << ebits) for m in range(1 << mbits)]
    return torch.tensor([x for x in v[:codes] if x <= top], dtype=torch.float32, device="cuda")


def _e2m1(x):
    """Real tensor -> E2M1 codes, nearest value, saturating."""
    v = _small_values(2, 1, 1, 8, 6.0)
    mag = torch.bucketize(x.abs(), (v[1:] + v[:-1]) / 2)
    return (mag + 8 * (x < 0)).to(torch.uint8)


def _words(fmt, x):
    """FP32 tensor -> raw words of an unscaled format."""
    if fmt == "fp64":
        return x.double().view(torch.int64)
    if fmt == "fp32":
        return x.view(torch.int32)
    if fmt == "tf32":
        return (x.view(torch.int32) + 0x1000) & ~0x1FFF
    if fmt in ("fp16", "bf16"):
        return x.to(torch.float16 if fmt == "fp16" else torch.bfloat16).view(torch.int16)
    if fmt in ("e4m3", "e5m2"):
        top, kind = (448.0, torch.float8_e4m3fn) if fmt == "e4m3" else (57344.0, torch.float8_e5m2)
        return x.clamp(-top, top).to(kind).view(torch.uint8)
    return _e2m1(x)


def _scaled(fmt, x):
    """FP32 matrix -> words and scale bytes of a block-scaled format (scale from the block's largest magnitude)."""
    kb = SCALE_BLOCK[fmt]
    blocks = x.view(x.shape[0], -1, kb)
    amax = blocks.abs().amax(2).clamp_min(2.0 ** -100)
    if fmt == "nvf4":
        sf = (amax / 6).clamp(2.0 ** -9, 448.0).to(torch.float8_e4m3fn)
        scale, sf = sf.float(), sf.view(torch.uint8)
    else:
        e = amax.log2().floor() - (8 if fmt == "mxe4m3" else 2)
        scale, sf = torch.exp2(e), (e + 127).clamp(0, 254).to(torch.uint8)
    q = (blocks / scale.unsqueeze(2)).view(x.shape)
    if fmt == "mxe4m3":
        return _words("e4m3", q), sf.contiguous()
    c = _e2m1(q)
    return (c[:, 0::2] | (c[:, 1::2] << 4)).contiguous(), sf.contiguous()


def _operand(case, rows, gen):
    fmt, K = case["fmt"], case["K"]
    if case.get("dist") == "exponents":         # random sign, exponent within +-20, random significand
        e = torch.randint(-20, 21, (rows, K), generator=gen, device="cuda") + 127
        m = torch.randint(0, 128, (rows, K), generator=gen, device="cuda")
        s = torch.randint(0, 2, (rows, K), generator=gen, device="cuda")
        return (((s << 15) | (e << 7) | m).to(torch.int32) & 0xFFFF).to(torch.int16), None, None
    x = torch.randn((rows, K), generator=gen, device="cuda")
    if fmt in SCALE_BLOCK:
        return (*_scaled(fmt, x), None)
    if fmt in ("e4m3", "e5m2", "e2m1"):         # per-row scales to the type's range, as FP8 GEMMs are fed
        s = x.abs().amax(1) / {"e4m3": 448.0, "e5m2": 57344.0, "e2m1": 6.0}[fmt]
        return _words(fmt, x / s.unsqueeze(1)), None, s
    return _words(fmt, x), None, None


def _probe_classes(case, A, B, gen):
    """Eight kinds of probe vectors in turn: plain values, outliers, subnormals, exact cancellation, one element of the
    largest exponent, ill-conditioned, infinities and NaNs, random bits."""
    n, K = A.shape
    eb, mb, low = {"fp16": (5, 10, 0), "bf16": (8, 7, 0), "tf32": (8, 10, 13), "e4m3": (4, 3, 0)}[case["fmt"]]
    exp = ((1 << eb) - 1) << (mb + low)
    big = exp - (1 << (mb + low))
    sign = 1 << (eb + mb + low)
    A, B = A.long(), B.long()
    k = torch.arange(n, device="cuda") % 8
    slot = torch.randint(0, K, (n, 1), generator=gen, device="cuda") == torch.arange(K, device="cuda")
    coin = torch.rand((n, K), generator=gen, device="cuda") < 0.5
    half = K // 2
    pick = lambda c: (k == c).unsqueeze(1)  # noqa: E731
    A = torch.where(pick(1) & slot, A + (3 << (mb + low)) * ((A & exp) < big - (4 << (mb + low))), A)
    A = torch.where(pick(2) & coin, A & ~exp, A)
    A2, B2 = torch.cat([A[:, :half]] * 2, 1), torch.cat([B[:, :half], B[:, :half] ^ sign], 1)
    A, B = torch.where(pick(3) | pick(5), A2, A), torch.where(pick(3) | pick(5), B2, B)
    A = torch.where(pick(5) & slot, A ^ (1 << low), A)
    A = torch.where(pick(4) & slot, (A & ~exp) | big, A)
    A = torch.where(pick(6) & slot & coin, torch.full_like(A, exp | (((1 << mb) - 1) << low if eb == 4 else 0)), A)
    A = torch.where(pick(7), torch.randint(0, 2 * sign, (n, K), generator=gen, device="cuda"), A)
    w = WORDS[BITS.get(case["fmt"], 8)]
    return A.to(w).contiguous(), B.to(w).contiguous()


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    M, N = case["M"], case["N"]
    state = {"op": case["op"], "K": case["K"], "model": mmasim.Model(case["arch"], case["fmt"], case["acc"])}
    if case["op"] == "dot":
        A, _, _ = _operand(case, M, gen)
        B, _, _ = _operand(case, M, gen)
        state["A"], state["B"] = _probe_classes(case, A, B, gen)
        state["C"] = torch.randn(M, generator=gen, device="cuda").view(torch.int32)
        return state
    state["A"], sfa, sa = _operand(case, M, gen)
    state["B"], sfb, sb = _operand(case, N, gen)
    c = None
    if case["c"]:
        c = torch.randn((M, N), generator=gen, device="cuda")
        c = c.double().view(torch.int64) if case["acc"] == "fp64" else _words(case["acc"], c)
    state["C"] = c
    kw = {}
    if sfa is not None:
        kw.update(sfa=sfa, sfb=sfb)
    if case.get("k_chunk"):
        kw["k_chunk"] = case["k_chunk"]
    if case.get("scales"):
        kw.update(row_scale=sa, col_scale=sb)
    state["kw"] = kw
    if case["op"] == "host":
        for name in ("A", "B", "C"):
            if state[name] is not None:
                host = torch.empty(state[name].shape, dtype=state[name].dtype, pin_memory=True)
                state[name] = host.copy_(state[name])
        state["out"] = torch.empty((M, N), dtype=WORDS[8 * ACC_BYTES[case["acc"]]], pin_memory=True)
    return state


def run(state):
    op, model = state["op"], state["model"]
    if op == "dot":
        return mmasim.dot_batch(model, state["A"], state["B"], state["C"])
    if op == "gemm":
        return mmasim.gemm(model, state["A"], state["B"], state["C"], K=state["K"], **state["kw"])
    if op == "accuracy":
        return accuracy.deviation_stats(model, state["A"], state["B"], state["C"])
    mmasim.gemm_host(model, state["A"], state["B"], state["C"], out=state["out"])
    return state["out"]


def work(case):
    M, N, K = case["M"], case["N"], case["K"]
    bits, acc = BITS.get(case["fmt"], 8), ACC_BYTES[case["acc"]]
    if case["op"] == "dot":
        return {"bytes": 2 * M * K * bits / 8 + 2 * M * acc, "flops": 2 * M * K}
    b = (M + N) * K * bits / 8 + M * N * acc * (2 if case["c"] else 1)
    if case["fmt"] in SCALE_BLOCK:
        b += (M + N) * K / SCALE_BLOCK[case["fmt"]]
    if case.get("scales"):
        b += 4 * (M + N)
    if case["op"] == "accuracy":                # the model's product and the FP64 product; eight sums come back
        return {"bytes": (M + N) * K * bits / 8 + (M * N * acc if case["c"] else 0) + 64, "flops": 4 * M * N * K}
    return {"bytes": b, "flops": 2 * M * N * K}


def tolerance(case):
    # the statistics are FP64 sums of up to 4 M deviations in no fixed order; the mean of signed ones cancels
    return {"rel": 1e-9} if case["op"] == "accuracy" else "exact"
