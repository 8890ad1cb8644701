"""FP16 products of few rows on the warp-level matrix instruction: against the generic kernels, bit for bit, at the edges of its tiles
(16 x 32 outputs), of its stages (128 elements of K) and of its ring of stages."""
import pytest
import torch

from test_gpu_tile_sizes import _inputs, gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("acc", ["fp32", "fp16"])
@pytest.mark.parametrize("M,N,K", [(1, 1, 8), (1, 33, 16), (16, 32, 112), (17, 31, 128), (15, 64, 144), (33, 100, 256), (3, 70, 1040), (16, 32, 2064)])
def test_few_rows_against_generic(M, N, K, acc):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model("hopper", "fp16", acc)
    for v in _inputs(("hopper", "fp16", acc), M, N, K, 700 + K):         # ordinary values, raw bit patterns, small magnitudes
        d = {k: gu.dev(x) for k, x in v.items()}
        forms = [dict(C=d["C"]), dict(C=None)]
        if acc == "fp32":
            forms.append(dict(C=d["C"], row_scale=torch.rand(M, device="cuda"), col_scale=torch.rand(N, device="cuda")))
        wide = [torch.nn.functional.pad(d[k], (0, 8))[:, :-8] for k in ("A", "B")]
        for kw in forms:
            want = mmasim.gemm(model, d["A"], d["B"], force_generic=True, **kw)
            for A, B in ((d["A"], d["B"]), wide):
                got = mmasim.gemm(model, A, B, **kw)
                assert mmasim.last_variant() == "matrix_instruction"
                assert torch.equal(got, want), ((M, N, K), list(kw), int((got != want).sum()))
