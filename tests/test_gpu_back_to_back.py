"""Calls one right behind the other: a kernel may be set up while the one before it ends, but reads nothing that is not finished and
overwrites nothing that is still read; outside and inside a captured graph, on one stream and on several threads' streams."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu
gu = pytest.importorskip("gpu_util") if torch.cuda.is_available() else None

# a kernel or a sequence of kernels each: small and large tiles, both matrix instructions (with the passes around them), dots, floating point
WORK = [(("hopper", "fp16", "fp32"), 16, 512, 512), (("hopper", "bf16", "fp32"), 512, 512, 512), (("ampere", "fp16", "fp32"), 300, 300, 256),
        (("hopper", "e4m3", "fp32"), 256, 1024, 256), (("cdna3", "bf16", "fp32"), 700, 700, 136), (("cdna1", "fp16", "fp32"), 700, 700, 128),
        (("cdna2", "fp16", "fp32"), 128, 128, 128), (("blackwell", "e4m3", "fp32"), 128, 256, 512), (("cdna1", "fp32", "fp32"), 64, 64, 64)]


def _operands():
    from paper_2511_10909_b200 import mmasim, workloads as wl
    out = []
    for n, (key, M, N, K) in enumerate(WORK):
        v = wl.normal_inputs(key[1], key[2], M, N, K, seed=800 + n)
        out.append((mmasim.Model(*key), *(gu.dev(v[k]) for k in ("A", "B", "C"))))
    return out


def _chain(operands):
    from paper_2511_10909_b200 import mmasim
    outs = []
    for model, A, B, C in operands:
        A2 = A.clone()                                  # written right before ...
        D = mmasim.gemm(model, A2, B, C)
        A2.zero_()                                      # ... and overwritten right behind
        E = mmasim.gemm(model, A, B, D)                 # C is what the call before wrote
        D.fill_(7)
        outs += [E, mmasim.gemm(model, A, B, E)]
    A, B, C = operands[2][1][:256, :32].contiguous(), operands[2][2][:256, :32].contiguous(), operands[2][3].reshape(-1)[:256].contiguous()
    d = mmasim.dot_batch(operands[2][0], A, B, C)
    outs.append(mmasim.dot_batch(operands[2][0], A, B, d))
    return outs


def _apart(operands):
    """The same with the GPU idle between any two kernels of different calls."""
    from paper_2511_10909_b200 import mmasim
    gemm, dots = mmasim.gemm, mmasim.dot_batch
    def alone(f):
        def call(*a, **kw):
            torch.cuda.synchronize()
            r = f(*a, **kw)
            torch.cuda.synchronize()
            return r
        return call
    mmasim.gemm, mmasim.dot_batch = alone(gemm), alone(dots)
    try:
        return _chain(operands)
    finally:
        mmasim.gemm, mmasim.dot_batch = gemm, dots


def test_calls_back_to_back():
    operands = _operands()
    want = _apart(operands)
    for _ in range(20):
        for got, w in zip(_chain(operands), want):
            assert torch.equal(got, w)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        _chain(operands)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        outs = _chain(operands)
    for _ in range(5):
        for x in outs:
            x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(outs, want))
    wrong = []
    def run():
        own = torch.cuda.Stream()
        with torch.cuda.stream(own):
            for _ in range(10):
                got = _chain(operands)
                own.synchronize()
                wrong.append(sum(not torch.equal(a, b) for a, b in zip(got, want)))
    threads = [threading.Thread(target=run) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert wrong == [0] * 30


def _products_only(operands, outs, sync=lambda: None):
    """Library calls and nothing else in the stream: D of one is C of the next, some in place; scratch of one call is that of the next
    (the large tiles' decoded operands, the matrix instruction's flags)."""
    from paper_2511_10909_b200 import mmasim
    for (model, A, B, C), (D, E) in zip(operands, outs):
        mmasim.gemm(model, A, B, C, out=D)
        sync()
        mmasim.gemm(model, A, B, D, out=E)
        sync()
        mmasim.gemm(model, A, B, E, out=E)
        sync()
        mmasim.gemm(model, A, B, E, out=D)
        sync()
    for (model, A, B, _), (D, E) in zip(reversed(operands), reversed(outs)):
        mmasim.gemm(model, A, B, D, out=D)
        sync()


def test_products_right_behind_each_other():
    operands = _operands()
    make = lambda: [tuple(torch.empty_like(C) for _ in range(2)) for _, _, _, C in operands]
    want = make()
    _products_only(operands, want, sync=torch.cuda.synchronize)
    same = lambda got: all(torch.equal(a, b) for x, y in zip(got, want) for a, b in zip(x, y))
    got = make()
    for _ in range(20):
        _products_only(operands, got)
        assert same(got)
    nodes = gu.recorded(lambda: _products_only(operands, got))[2]
    assert "other" not in nodes and all(x in ("alloc", "free") or "mmasim" in x for x in nodes), nodes
    stream = torch.cuda.Stream()
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        _products_only(operands, got)
    for _ in range(5):
        for x in got:
            x[0].zero_(), x[1].zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert same(got)
    wrong = []
    def run():
        own, mine = torch.cuda.Stream(), make()
        with torch.cuda.stream(own):
            for _ in range(10):
                _products_only(operands, mine)
                own.synchronize()
                wrong.append(not same(mine))
    torch.cuda.synchronize()
    threads = [threading.Thread(target=run) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert wrong == [False] * 30
