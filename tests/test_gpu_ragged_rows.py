"""Large tiles over rows that are no whole number of chunks of 32, or that start off 16 bytes: against the generic kernels, bit for bit."""
import pytest
import torch

from test_gpu_tile_sizes import KEYS, _inputs, gu

pytestmark = pytest.mark.gpu


# one block and its neighbours of a chunk; a tile of every size less one row, whole, and one row more
@pytest.mark.parametrize("M,N,blocks", [(1, 1, 1), (63, 129, 3), (128, 64, 5), (129, 65, 9)])
@pytest.mark.parametrize("key", [k for k in KEYS if not k[1].startswith("mx")], ids=lambda k: "-".join(k))
def test_ragged_rows_against_generic(key, M, N, blocks):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    K = model.l_max * blocks
    for v in _inputs(key, M, N, K, 600 + blocks):           # ordinary values, raw bit patterns, small magnitudes
        v["C"][::3, ::2] = 0x8000 if key[2] == "fp16" else 0x80000000         # -0
        d = {k: gu.dev(x) for k, x in v.items()}
        want = mmasim.gemm(model, d["A"], d["B"], d["C"], force_generic=True)
        for A, B in ((d["A"], d["B"]), [torch.nn.functional.pad(d[k], (0, 3))[:, :-3] for k in ("A", "B")]):
            got = mmasim.gemm(model, A, B, d["C"], large_tiles=True)
            assert mmasim.last_variant() == "large_tiles"
            assert torch.equal(got, want), (key, (M, N, K), int((got != want).sum()))


# rows off 16 bytes under scale factors, and with promoted sums and dequantisation scales: every kernel that takes either
@pytest.mark.parametrize("key", [k for k in KEYS if k[2] == "fp32" and (k[1].startswith("mx") or not k[0].startswith("cdna"))], ids=lambda k: "-".join(k))
def test_strides_off_16_bytes_with_scales_and_promotion(key):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    for M, N, K in ((63, 129, 192), (130, 65, 384)):
        scales = dict(row_scale=torch.rand(M, device="cuda") * 4, col_scale=torch.rand(N, device="cuda") * 4)
        for v in _inputs(key, M, N, K, 660 + M):
            d = {k: gu.dev(x) for k, x in v.items()}
            sf = {k: d[k] for k in ("sfa", "sfb") if k in d}
            A, B = (torch.nn.functional.pad(d[k], (0, 3))[:, :-3] for k in ("A", "B"))
            for kw in ({}, dict(k_chunk=32), dict(k_chunk=64, **scales), dict(k_chunk=K, **scales)):
                want = mmasim.gemm(model, d["A"], d["B"], d["C"], force_generic=True, **kw, **sf)
                got = mmasim.gemm(model, A, B, d["C"], large_tiles=True, **kw, **sf)
                assert mmasim.last_variant() == "large_tiles"
                assert torch.equal(got, want), (key, (M, N, K), list(kw), int((got != want).sum()))


@pytest.mark.parametrize("key", [("ampere", "fp16", "fp32"), ("hopper", "e4m3", "fp32"), ("cdna1", "bf16", "fp32")], ids="-".join)
def test_graphs_of_ragged_calls_hold_no_memory(key):
    """What is recorded can be cloned and instantiated twice, as a graph with memory nodes cannot."""
    from cuda.bindings import runtime
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    M, N, K = 1000, 1111, 96 + model.l_max if model.l_max < 32 else 128
    v = _inputs(key, M, N, K, 650)[0]
    A, B, C = (gu.dev(v[k]) for k in ("A", "B", "C"))
    A = torch.nn.functional.pad(A, (0, 3))[:, :-3]
    want = mmasim.gemm(model, A, B, C, large_tiles=True)
    assert mmasim.last_variant() == "large_tiles"
    graph, out, nodes = gu.recorded(lambda: mmasim.gemm(model, A, B, C, large_tiles=True))
    assert len(nodes) == 1 and "direct_kernel" in nodes[0], nodes
    done = lambda r: (r[0] == runtime.cudaError_t.cudaSuccess or pytest.fail(str(r[0]))) and r[-1]
    raw = runtime.cudaGraph_t(graph.raw_cuda_graph())
    execs = [done(runtime.cudaGraphInstantiate(g, 0)) for g in (raw, raw, done(runtime.cudaGraphClone(raw)))]
    for e in execs:
        out.zero_()
        done(runtime.cudaGraphLaunch(e, torch.cuda.current_stream().cuda_stream) + (True,))
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        done(runtime.cudaGraphExecDestroy(e) + (True,))
