"""The floating-point kernels (Phi_FMA in FP32 and FP64, Phi_FTZ-AddMul) in both tile sizes at ragged K and odd row strides, against the
generic kernels, bit for bit; -0 accumulators and products (the filling of the last chunk must not turn them into +0)."""
import numpy as np
import pytest
import torch

from paper_2511_10909_b200 import workloads as wl

pytestmark = pytest.mark.gpu
gu = pytest.importorskip("gpu_util") if torch.cuda.is_available() else None


@pytest.mark.parametrize("key", [("hopper", "fp64", "fp64"), ("cdna1", "fp32", "fp32"), ("cdna2", "fp16", "fp32"), ("cdna2", "bf16", "fp32"),
                                 ("cdna2", "bf16_1k", "fp32")], ids=lambda k: "-".join(k))
def test_any_k_and_stride(key):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    unit = model.P or 1
    for n, (M, N, K) in enumerate([(1, 1, 1), (33, 65, 5), (31, 64, 17), (34, 70, 64), (130, 129, 35), (370, 430, 35), (700, 1300, 36), (1290, 1300, 52)]):
        K = -(-K // unit) * unit
        g = wl.rng(60 + n)
        inp = wl.normal_inputs(key[1], key[2], M, N, K, seed=n)
        wild = {k: g.integers(0, 1 << 8 * x.dtype.itemsize - 1, x.shape, dtype=np.uint64).astype(x.dtype) * 2 + g.integers(0, 2, x.shape).astype(x.dtype)
                for k, x in inp.items()}
        minus = {k: np.full_like(x, 1 << (8 * x.dtype.itemsize - 1)) if k != "B" else np.abs(x) * 0 for k, x in inp.items()}
        for v in (inp, wild, minus):
            A, B, C = (gu.dev(v[k]) for k in ("A", "B", "C"))
            for c in (C, None):
                want = mmasim.gemm(model, A, B, c, force_generic=True)
                assert torch.equal(mmasim.gemm(model, A, B, c), want), (key, (M, N, K), c is None)
                strided = [torch.nn.functional.pad(x, (0, p))[:, :-p] for x, p in ((A, 1), (B, 2))]
                assert torch.equal(mmasim.gemm(model, *strided, c), want), (key, (M, N, K), "strided")
                # few tiles of 16 x 16 per SM stay with the generic kernels, unless K and the rows suit the others
                assert (mmasim.last_variant() == "generic") == (key[2] == "fp32" and M * N < 150 * 150), (key, (M, N, K), mmasim.last_variant())


@pytest.mark.parametrize("fmt", ["fp16", "bf16", "tf32", "fp32", "e4m3", "e5m2"])
def test_reference_fp64_against_widened_operands(fmt):
    from paper_2511_10909_b200 import accuracy, mmasim
    model = mmasim.Model("cdna1" if fmt == "fp32" else "hopper", fmt, "fp32")
    for M, N, K in ((3, 5, 64), (130, 70, 96)):
        A, B, C = (gu.dev(wl.normal_inputs(fmt, "fp32", M, N, K, seed=7)[k]) for k in ("A", "B", "C"))
        for c in (C, None):
            assert torch.equal(mmasim.reference_fp64(model, A, B, c), accuracy.reference_fp64(fmt, "fp32", A, B, c))
