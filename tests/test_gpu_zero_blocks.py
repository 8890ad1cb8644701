"""Blocks without a nonzero product in the large-tile kernels (exponent maximum on the tensor cores, range test left out): the result is the
accumulator, whatever its size.  Tiles of 64 x 64 with remainders, against the generic kernel, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2511_10909_b200 import workloads as wl

pytestmark = pytest.mark.gpu
gu = pytest.importorskip("gpu_util") if torch.cuda.is_available() else None


@pytest.mark.parametrize("c_exp", [0, -29, -30, -31, -53, -100, -126, -149, 101])
@pytest.mark.parametrize("arch, fmt", [("ampere", "fp16"), ("turing", "fp16"), ("ampere", "bf16")])
def test_zero_blocks(arch, fmt, c_exp):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(arch, fmt, "fp32")
    for M, N, K in ((64, 64, 32), (65, 130, 96), (129, 63, 256)):
        g = wl.rng(11)
        x, y = (g.standard_normal((r, K)) * 2.0 ** -g.integers(0, 15, (r, K)) for r in (M, N))
        x *= np.repeat(g.random((M, K // 8)) < 0.5, 8, axis=1)          # half of the blocks of 8 are zero, of either sign
        y *= g.random((N, K)) < 0.8
        c = (g.standard_normal((M, N)) * 2.0 ** c_exp).astype(np.float32)
        A, B = (torch.from_numpy(wl.cast(v.astype(np.float32), fmt).view(np.int16)).cuda() for v in (x, y))
        C = torch.from_numpy(c.view(np.int32)).cuda()
        got = mmasim.gemm(model, A, B, C, large_tiles=True)
        want = mmasim.gemm(model, A, B, C, force_generic=True)
        assert torch.equal(got, want), (M, N, K, int((got != want).sum()))
