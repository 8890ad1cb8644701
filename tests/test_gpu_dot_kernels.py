"""The streaming kernels of dot_batch against the generic arithmetic, bit for bit: every row length they stage (4 to 128 bytes) or read
directly, an odd number of dots (a last tile that ends inside a 16-byte chunk), one dot, chains of several blocks."""
import numpy as np
import pytest
import torch

from paper_2511_10909_b200 import workloads as wl

pytestmark = pytest.mark.gpu
gu = pytest.importorskip("gpu_util") if torch.cuda.is_available() else None

KEYS = [("hopper", "e4m3", "fp32"), ("hopper", "e5m2", "fp16"), ("ada", "e4m3", "fp32"), ("ada", "e5m2", "fp16"), ("blackwell", "e4m3", "fp32"),
        ("blackwell", "e5m2", "fp16"), ("cdna3", "fp16", "fp32"), ("cdna3", "bf16", "fp32"), ("cdna3", "tf32", "fp32"),
        ("volta", "fp16", "fp32"), ("hopper", "fp16", "fp32"), ("hopper", "fp16", "fp16"), ("ampere", "bf16", "fp32"), ("hopper", "tf32", "fp32")]


@pytest.mark.parametrize("key", KEYS, ids=lambda k: "-".join(k))
def test_dots_against_generic(key):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    g = wl.rng(41)
    for K in (4, 8, 16, 32, 64, 96, 128):
        if K > model.l_max and K % model.l_max:
            continue
        for n in (1, 261):
            inp = wl.normal_inputs(key[1], key[2], n, n, K, seed=K + n)
            inp["A"][g.random(inp["A"].shape) < 0.1] = 0
            wild = {k: g.integers(0, 1 << 8 * x.dtype.itemsize, x.shape, dtype=np.uint64).astype(x.dtype) for k, x in inp.items()}
            low = {k: x & ~x.dtype.type(1 << (8 * x.dtype.itemsize - 2)) for k, x in wild.items()}
            zero = dict(wild, A=np.where(g.random((n, 1)) < 0.5, wild["A"], 0).astype(wild["A"].dtype))
            for v in (inp, wild, low, zero):
                A, B, C = (gu.dev(v[k]) for k in ("A", "B", "C"))
                for c in (C, None):
                    want = torch.diagonal(mmasim.gemm(model, A, B, c, force_generic=True))
                    got = mmasim.dot_batch(model, A, B, None if c is None else torch.diagonal(c).contiguous())
                    assert mmasim.last_kernel() in ("dot_tfdpa", "dot_trfdpa")
                    assert torch.equal(got, want), (key, K, n, c is None, int((got != want).sum()))
