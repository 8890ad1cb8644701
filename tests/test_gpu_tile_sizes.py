"""Every tile size of the FDPA kernels at the edges of tiles, chunks and blocks: the small-tile kernels (8 x 16, 16 x 16 and
32 x 32 outputs, any K, any row stride) and the large-tile kernels, each against the generic kernels, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2511_10909_b200 import workloads as wl

pytestmark = pytest.mark.gpu
gu = pytest.importorskip("gpu_util") if torch.cuda.is_available() else None

# one row per instantiation: element kind, block length, rho, family
KEYS = [("volta", "fp16", "fp32"), ("volta", "fp16", "fp16"), ("ampere", "fp16", "fp32"), ("ampere", "fp16", "fp16"), ("hopper", "fp16", "fp32"),
        ("hopper", "fp16", "fp16"), ("ampere", "bf16", "fp32"), ("hopper", "bf16", "fp32"), ("ampere", "tf32", "fp32"), ("hopper", "tf32", "fp32"),
        ("ada", "e4m3", "fp32"), ("ada", "e5m2", "fp16"), ("hopper", "e4m3", "fp32"), ("hopper", "e5m2", "fp16"), ("blackwell", "e4m3", "fp32"),
        ("blackwell", "e5m2", "fp32"), ("blackwell", "e3m2", "fp16"), ("blackwell", "e2m3", "fp32"), ("blackwell", "e2m1", "fp32"),
        ("blackwell", "mxe4m3", "fp32"), ("blackwell", "mxe2m1", "fp32"), ("cdna3", "bf16", "fp32"), ("cdna3", "fp16", "fp32"),
        ("cdna3", "tf32", "fp32"), ("cdna3", "e5m2", "fp32"), ("cdna1", "fp16", "fp32"), ("cdna1", "bf16", "fp32")]
# M, N, blocks of K: one output, a tile and one more in each size, one block, a chunk less and more a block
SHAPES = [(1, 1, 1), (8, 16, 3), (9, 17, 9), (17, 33, 5), (300, 200, 7), (700, 500, 3)]


def _wild(g, x, width):
    n = x.dtype.itemsize
    if n == 1:
        return g.integers(0, 1 << width, x.shape, dtype=np.uint8)
    return (g.integers(0, 1 << (8 * n - 1), x.shape, dtype=np.uint64) * 2 + g.integers(0, 2, x.shape, dtype=np.uint64)).astype(x.dtype)


def _inputs(key, M, N, K, seed):
    """Ordinary values with zeros, raw bit patterns, and bit patterns of small magnitude."""
    g = wl.rng(seed)
    inp = wl.normal_inputs(key[1], key[2], M, N, -(-K // 32) * 32 if key[1].startswith("mx") else K, seed=seed)
    inp["A"][g.random(inp["A"].shape) < 0.1] = 0
    inp["C"][g.random(inp["C"].shape) < 0.2] = 0
    width = {"e2m1": 4, "e2m3": 6, "e3m2": 6}.get(key[1].replace("mx", ""), 8)
    wild = {k: _wild(g, inp[k], width) for k in ("A", "B", "C")}
    for k in ("sfa", "sfb"):
        if k in inp:
            wild[k] = g.integers(0, 256, inp[k].shape, dtype=np.uint8)
    small = dict(wild)
    for k in ("A", "B", "C"):
        bits = width if wild[k].dtype.itemsize == 1 else 8 * wild[k].dtype.itemsize
        small[k] = wild[k] & ~wild[k].dtype.type(1 << (bits - 2))
    return [inp, wild, small]


@pytest.mark.parametrize("key", KEYS, ids=lambda k: "-".join(k))
def test_tile_sizes_against_generic(key):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    unit = 32 if key[1].startswith("mx") else model.l_max
    for n, (M, N, blocks) in enumerate(SHAPES):
        K = unit * blocks
        for v in _inputs(key, M, N, K, 100 + n):
            d = {k: gu.dev(x) for k, x in v.items()}
            sf = {k: d[k] for k in ("sfa", "sfb") if k in d}
            forms = [{}]
            if key[2] == "fp32" and model.family in ("t", "st") and blocks % 3 == 0:
                forms.append({"k_chunk": 3 * unit if blocks > 3 else unit})
            for kw in forms:
                want = mmasim.gemm(model, d["A"], d["B"], d["C"], force_generic=True, **kw, **sf)
                got = mmasim.gemm(model, d["A"], d["B"], d["C"], **kw, **sf)
                assert torch.equal(got, want), (key, (M, N, K), kw, int((got != want).sum()))
                # rows at odd addresses: one word between the rows of A and of B
                strided = [torch.nn.functional.pad(d[k], (0, 1))[:, :-1] for k in ("A", "B")]
                got = mmasim.gemm(model, *strided, d["C"], **kw, **sf)
                assert torch.equal(got, want), (key, (M, N, K), kw, "strided", int((got != want).sum()))


@pytest.mark.parametrize("key", KEYS, ids=lambda k: "-".join(k))
def test_large_tiles_against_generic(key):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    for n, (M, N, K) in enumerate([(1, 1, 32), (128, 64, 64), (129, 65, 96), (200, 300, 160)]):
        for v in _inputs(key, M, N, K, 200 + n):
            d = {k: gu.dev(x) for k, x in v.items()}
            sf = {k: d[k] for k in ("sfa", "sfb") if k in d}
            forms = [{}]
            if key[2] == "fp32" and model.family in ("t", "st"):
                forms.append({"k_chunk": 32})
            for kw in forms:
                want = mmasim.gemm(model, d["A"], d["B"], d["C"], force_generic=True, **kw, **sf)
                got = mmasim.gemm(model, d["A"], d["B"], d["C"], large_tiles=True, **kw, **sf)
                assert torch.equal(got, want), (key, (M, N, K), kw, int((got != want).sum()))


@pytest.mark.parametrize("key", [("blackwell", "mxf4", "fp32"), ("rtx_blackwell", "nvf4", "fp32")], ids=lambda k: "-".join(k))
def test_group_scaled_rows_against_generic(key):
    """The kernel that emulates the group-scaled rows, which otherwise only runs behind the matrix instruction (MXFP4) or not at all."""
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    for n, (M, N, K) in enumerate([(1, 1, 64), (128, 64, 128), (129, 65, 192), (200, 300, 320)]):
        for v in _inputs(key, M, N, K, 500 + n):
            d = {k: gu.dev(x) for k, x in v.items()}
            sf = {k: d[k] for k in ("sfa", "sfb")}
            for c in (d["C"], None):
                want = mmasim.gemm(model, d["A"], d["B"], c, K=K, force_generic=True, **sf)
                got = mmasim.gemm(model, d["A"], d["B"], c, K=K, large_tiles=True, **sf)
                assert mmasim.last_kernel() == "gstfdpa" and mmasim.last_variant() == "large_tiles"
                assert torch.equal(got, want), (key, (M, N, K), c is None, int((got != want).sum()))


@pytest.mark.parametrize("key", KEYS, ids=lambda k: "-".join(k))
def test_special_values_among_others(key):
    """A few infinities, NaNs, zeros opposite them and huge values (overflow before and after a special value of the same chunk) in whole
    and partial chunks, and E-FDPA sums that no double holds: from a few rows to all of them."""
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    unit = 32 if key[1].startswith("mx") else model.l_max
    for n, (M, N, K, share) in enumerate([(40, 70, 256, 0.001), (100, 130, 160 + unit % 32, 0.004), (500, 600, 96, 0.02)]):
        g = wl.rng(400 + n)
        v = wl.normal_inputs(key[1], key[2], M, N, -(-K // 32) * 32, seed=400 + n)
        for k in ("A", "B"):
            v[k] = v[k][:, :K].copy()
            size = v[k].dtype.itemsize
            width = {"e2m1": 4, "e2m3": 6, "e3m2": 6}.get(key[1].replace("mx", ""), 8) if size == 1 else 8 * size
            top = ((1 << (width - 1)) - 1) if size < 4 else 0x7FFFE000
            exps = {"fp16": 0x7C00, "bf16": 0x7F80, "tf32": 0x7F800000}.get(key[1], 0x7C if "e5m2" in key[1] else top)
            for word in (exps, top, 0, exps - (1 << 13 if size == 4 else 1)):        # infinity (or the largest pattern), NaN, zero, the largest number
                at = g.random(v[k].shape) < share
                v[k][at] = (word | (g.integers(0, 2, int(at.sum())) << (width - 1))).astype(v[k].dtype)
        if model.family == "e":
            v["C"][::2] = (v["C"][::2] & np.uint32(0x807FFFFF)) | np.uint32(0x08000000)      # far below the products
        d = {k: gu.dev(x) for k, x in v.items()}
        sf = {k: d[k] for k in ("sfa", "sfb") if k in d}
        want = mmasim.gemm(model, d["A"], d["B"], d["C"], force_generic=True, **sf)
        got = mmasim.gemm(model, d["A"], d["B"], d["C"], **sf)
        assert torch.equal(got, want), (key, (M, N, K), int((got != want).sum()))
        if key[2] == "fp32" and model.family in ("t", "st"):
            for kc in {unit, K} if K % unit == 0 else {K}:
                want = mmasim.gemm(model, d["A"], d["B"], d["C"], force_generic=True, k_chunk=kc, **sf)
                got = mmasim.gemm(model, d["A"], d["B"], d["C"], k_chunk=kc, **sf)
                assert torch.equal(got, want), (key, (M, N, K), kc, int((got != want).sum()))
