"""The number of kernels that the benchmark says a call launches, against the kernels of the call recorded into a graph."""
import pytest
import torch

from paper_2511_10909_b200 import workloads as wl

pytestmark = pytest.mark.gpu
gu = pytest.importorskip("gpu_util") if torch.cuda.is_available() else None


@pytest.mark.parametrize("key,large", [(("hopper", "e4m3", "fp32"), False), (("hopper", "e4m3", "fp32"), True), (("ada", "e5m2", "fp16"), True), (("volta", "fp16", "fp32"), True),
                                       (("ampere", "bf16", "fp32"), True), (("ampere", "tf32", "fp32"), True), (("blackwell", "mxe4m3", "fp32"), True), (("cdna3", "bf16", "fp32"), True),
                                       (("cdna3", "e4m3", "fp32"), True), (("cdna1", "fp16", "fp32"), True), (("hopper", "fp16", "fp32"), False), (("hopper", "bf16", "fp32"), False),
                                       (("hopper", "tf32", "fp32"), False), (("blackwell", "e4m3", "fp32"), False), (("blackwell", "e2m1", "fp32"), False), (("blackwell", "mxe4m3", "fp32"), False),
                                       (("blackwell", "mxe2m3", "fp32"), False), (("blackwell", "mxf4", "fp32"), False), (("blackwell", "nvf4", "fp32"), False), (("cdna2", "fp16", "fp32"), False),
                                       (("cdna1", "fp32", "fp32"), False), (("hopper", "fp64", "fp64"), False)], ids=str)
def test_kernels_per_call(key, large):
    import bench
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    M = N = K = 512
    d = {k: gu.dev(x) for k, x in wl.normal_inputs(key[1], key[2], M, N, K, seed=90).items()}
    call = lambda: mmasim.gemm(model, d["A"], d["B"], d["C"], K=K, large_tiles=large, **{k: d[k] for k in ("sfa", "sfb") if k in d})
    call()
    kernel, variant = mmasim.last_kernel(), mmasim.last_variant()
    kernels = [x for x in gu.recorded(call)[2] if "mmasim" in x]
    assert len(kernels) == bench.kernels_per_call(kernel, variant, model), (key, kernel, variant, kernels)
    assert not large or variant == "large_tiles"
