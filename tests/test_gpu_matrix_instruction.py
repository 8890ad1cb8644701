"""The rows that run on the B200's own matrix instruction, against the generic kernels' integer arithmetic, bit for bit: at the edges of
tiles (16 to 256 rows of A by 128 rows of B), of stages (128 bytes of K) and of the ring of stages, with more tiles than SMs (both
accumulators and every barrier phase), blocks shorter than the instruction's, the dequantisation epilogue, and products around and
below 2^-126, where the instruction and the model part and the emulation has to take over."""
import numpy as np
import pytest
import torch

from paper_2511_10909_b200 import workloads as wl

pytestmark = pytest.mark.gpu
gu = pytest.importorskip("gpu_util") if torch.cuda.is_available() else None

# one row per instruction kind, operand packing and accumulator
KEYS = [("hopper", "fp16", "fp32"), ("hopper", "fp16", "fp16"), ("rtx_blackwell", "bf16", "fp32"), ("hopper", "tf32", "fp32"),
        ("blackwell", "e4m3", "fp32"), ("blackwell", "e5m2", "fp16"), ("blackwell", "e3m2", "fp32"), ("blackwell", "e2m3", "fp16"),
        ("blackwell", "e2m1", "fp32"), ("blackwell", "mxe4m3", "fp32"), ("blackwell", "mxe2m3", "fp32"), ("blackwell", "mxe2m1", "fp32"),
        ("blackwell", "mxf4", "fp32"), ("rtx_blackwell", "nvf4", "fp32")]
# M, N, blocks of K
SHAPES = [(1, 1, 1), (16, 128, 4), (17, 129, 5), (129, 127, 33), (257, 300, 18), (2500, 1200, 3)]


def _bits(g, x, width):
    n = x.dtype.itemsize
    return g.integers(0, 1 << (width if n == 1 else 8 * n), x.shape, dtype=np.uint64).astype(x.dtype)


def _width(key):
    return {"e2m1": 4, "e2m3": 6, "e3m2": 6}.get(key[1].replace("mx", ""), 8)


def _variants(key, M, N, K, seed):
    """Ordinary values with zeros, raw bit patterns, and bit patterns whose magnitudes (or scale factors) stay small."""
    g = wl.rng(seed)
    inp = wl.normal_inputs(key[1], key[2], M, N, K, seed=seed)
    inp["A"][g.random(inp["A"].shape) < 0.1] = 0
    inp["C"][g.random(inp["C"].shape) < 0.2] = 0
    width = _width(key)
    wild = {k: _bits(g, inp[k], width) for k in ("A", "B", "C")}
    small = {k: wild[k] & ~wild[k].dtype.type(1 << ((width if wild[k].dtype.itemsize == 1 else 8 * wild[k].dtype.itemsize) - 2))
             for k in ("A", "B", "C")}
    for k in ("sfa", "sfb"):
        if k in inp:
            wild[k] = g.integers(0, 256, inp[k].shape, dtype=np.uint8)
            small[k] = g.integers(0, 128, inp[k].shape, dtype=np.uint8)
    return [inp, wild, small]


# kinds with products below 2^-126, which small calls leave to the emulation
GUARDED = ("bf16", "tf32", "mxe4m3", "mxe5m2", "mxe2m3", "mxe3m2", "mxe2m1")


def _compare(model, v, K, C, what, ran=True, **kw):
    """`ran`: the matrix instruction has to be what computes it."""
    from paper_2511_10909_b200 import mmasim
    d = {k: gu.dev(x) for k, x in v.items()}
    sf = {k: d[k] for k in ("sfa", "sfb") if k in d}
    c = None if C is None else gu.dev(C)
    want = mmasim.gemm(model, d["A"], d["B"], c, K=K, force_generic=True, **kw, **sf)
    got = mmasim.gemm(model, d["A"], d["B"], c, K=K, **kw, **sf)
    assert not ran or mmasim.last_variant() == "matrix_instruction", (what, mmasim.last_variant())
    assert torch.equal(got, want), (what, int((got != want).sum()))


@pytest.mark.parametrize("key", KEYS, ids=lambda k: "-".join(k))
def test_matrix_instruction_against_generic(key):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    for n, (M, N, blocks) in enumerate(SHAPES):
        K = model.l_max * blocks
        for v in _variants(key, M, N, K, 300 + n):
            for C in (v["C"], None):
                _compare(model, v, K, C, (key, (M, N, K), C is None), ran=key[1] not in GUARDED or M >= 1000)
    assert mmasim.copy_timeouts() == 0


@pytest.mark.parametrize("acc", ["fp32", "fp16"])
def test_fp16_on_either_instruction(acc):
    """FP16 products of at most 296 tiles of 16 x 32 run on mma.sync, which leaves most of the shapes above to it; larger ones on tcgen05.mma:
    every width of its tiles, K beyond its ring of stages and off a stage, short blocks, the dequantisation epilogue."""
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model("hopper", "fp16", acc)
    g = wl.rng(340)
    for n, (M, N, K) in enumerate([(16, 9472, 48), (16, 9473, 48), (1, 9600, 1040), (17, 5000, 2064), (40, 4000, 144), (70, 3000, 1040), (129, 1100, 528), (300, 1000, 2064),
                                   (50, 2400, 8)]):
        tiles = -(-M // 16) * -(-N // 32)
        kws = [{}] if acc == "fp16" else [{}, dict(row_scale=gu.dev(g.standard_normal(M).astype(np.float32)), col_scale=gu.dev(g.standard_normal(N).astype(np.float32)))]
        for v in _variants(("hopper", "fp16", acc), M, N, K, 341 + n):
            for kw in kws:
                for C in (v["C"], None):
                    _compare(model, v, K, C, (acc, (M, N, K), list(kw), C is None), **kw)
        A, B = gu.dev(v["A"]), gu.dev(v["B"])
        nodes = gu.recorded(lambda: mmasim.gemm(model, A, B))[2]
        ran = [x for x in nodes if "mma_kernel" in x]
        assert len(ran) == 1 and ("warp_mma_kernel" in ran[0]) == (tiles <= 296) and ("umma_kernel" in ran[0]) == (tiles > 296), ((M, N, K), nodes)
    assert mmasim.copy_timeouts() == 0


@pytest.mark.parametrize("key", [k for k in KEYS if k[1] in GUARDED], ids=lambda k: "-".join(k))
def test_few_rows_of_kinds_with_small_products(key):
    """Every width of tile (16 to 256 rows of A) with K long enough that the instruction runs; flags at the edges of such tiles."""
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    for n, (M, N) in enumerate([(1, 300), (16, 129), (17, 257), (33, 140), (70, 300), (131, 390), (300, 700)]):
        K = 4096 if M < 100 else 1024
        for v in _variants(key, M, N, K, 310 + n):
            _compare(model, v, K, v["C"], (key, (M, N, K)))


@pytest.mark.parametrize("key", [("blackwell", "mxe4m3", "fp32"), ("blackwell", "mxf4", "fp32"), ("blackwell", "nvf4", "fp32")],
                         ids=lambda k: "-".join(k))
def test_scale_factors_round_the_ring(key):
    """Every stage's columns of scale factors are written over many times, by values that differ from block to block: long K, more tiles
    than SMs."""
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    for n, (M, N, K) in enumerate([(20, 2400, 8192), (300, 150, 16384), (1500, 2000, 2048)]):
        v = wl.normal_inputs(key[1], key[2], M, N, K, seed=320 + n)
        g = wl.rng(321 + n)
        lo, hi = (40, 72) if key[1] == "nvf4" else (112, 132)
        for k in ("sfa", "sfb"):
            v[k] = g.integers(lo, hi, v[k].shape, dtype=np.uint8)
        _compare(model, v, K, v["C"], (key, (M, N, K)))
    assert mmasim.copy_timeouts() == 0


@pytest.mark.parametrize("key,K", [(("hopper", "fp16", "fp32"), 8), (("blackwell", "e4m3", "fp32"), 16), (("blackwell", "mxe4m3", "fp32"), 16),
                                   (("blackwell", "mxf4", "fp32"), 32), (("blackwell", "nvf4", "fp32"), 32)], ids=str)
def test_block_shorter_than_the_instruction_and_dequantisation(key, K):
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    g = wl.rng(31)
    M, N = 50, 140
    rs, cs = (gu.dev(g.standard_normal(n).astype(np.float32)) for n in (M, N))
    for v in _variants(key, M, N, -(-K // 32) * 32, 330):
        for kw in ({}, dict(row_scale=rs, col_scale=cs)):
            _compare(model, v, K, v["C"], (key, K, list(kw)), ran=key[1] not in GUARDED + ("mxf4",), **kw)


@pytest.mark.parametrize("key", [("hopper", "bf16", "fp32"), ("hopper", "tf32", "fp32"), ("blackwell", "mxe4m3", "fp32"),
                                 ("blackwell", "mxe5m2", "fp32"), ("blackwell", "mxe2m1", "fp32"), ("blackwell", "mxf4", "fp32")],
                         ids=lambda k: "-".join(k))
def test_products_below_the_smallest_normal(key):
    """Exponent sums from far below -126 to just above, zero and nonzero accumulators; large enough that the matrix instruction runs."""
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    M, N, K = 1100, 1000, 4 * model.l_max
    for n, centre in enumerate((-170, -156, -144, -132, -126, -120, -112, -104, -90)):
        g = wl.rng(350 + n)
        v = {k: x for k, x in wl.normal_inputs(key[1], key[2], M, N, K, seed=n).items()}
        if key[1] in ("bf16", "tf32"):
            for k in ("A", "B"):
                low = 7 if key[1] == "bf16" else 23
                e = np.clip(127 + centre // 2 + g.integers(-6, 7, v[k].shape), 0, 254)
                v[k] = ((_bits(g, v[k], 8).astype(np.int64) & ~(255 << low)) | (e << low)).astype(v[k].dtype)
        else:
            for k, s in (("A", "sfa"), ("B", "sfb")):
                v[k] = _bits(g, v[k], _width(key))
                if key[1] == "mxe4m3":
                    v[k][(v[k] & 0x7F) == 0x7F] = 0
                if key[1] == "mxe5m2":
                    v[k][(v[k] & 0x7C) == 0x7C] = 0
                v[s] = np.clip(127 + centre // 2 + g.integers(-3, 4, v[s].shape), 0, 254).astype(np.uint8)
        near = (g.integers(0, 2, (M, N)) << 31) | (np.clip(centre + 127 + g.integers(-9, 9, (M, N)), 0, 254) << 23) | g.integers(0, 1 << 23, (M, N))
        for C in (None, near.astype(np.uint32), np.where(g.random((M, N)) < 0.5, 0, 0x80000001).astype(np.uint32)):
            _compare(model, v, K, C, (key, centre, C is None))


@pytest.mark.parametrize("key", [("blackwell", "mxe4m3", "fp32"), ("blackwell", "mxe5m2", "fp32"), ("blackwell", "mxe3m2", "fp32"),
                                 ("rtx_blackwell", "mxe2m1", "fp32"), ("blackwell", "mxf4", "fp32")], ids=lambda k: "-".join(k))
def test_zero_blocks_under_small_scale_factors(key):
    """Blocks of zeros (of either sign, and with the unused bits of a code set) under the smallest and under arbitrary small factors, beside
    blocks that are zero but for one element: the first flag nothing, the last do."""
    from paper_2511_10909_b200 import mmasim
    model = mmasim.Model(*key)
    packed = key[1] == "mxf4"
    per = 16 if packed else 32
    sign = 0x88 if packed else 1 << (_width(key) - 1)
    junk = 0 if packed else 0xFF & ~((1 << _width(key)) - 1)
    for n, (M, N, K) in enumerate([(900, 800, 64), (515, 520, 1024), (130, 2500, 4096)]):
        g = wl.rng(380 + n)
        v = wl.normal_inputs(key[1], key[2], M, N, K, seed=380 + n)
        for k, s in (("A", "sfa"), ("B", "sfb")):
            blocks = v[k].reshape(v[k].shape[0], -1, per)
            zero = g.random(blocks.shape[:2]) < 0.1
            blocks[zero] = g.choice(np.array([0, sign, junk, sign | junk], dtype=np.uint8), (int(zero.sum()), per))
            v[s] = np.where(zero, np.where(g.random(zero.shape) < 0.5, 0, g.integers(0, 80, zero.shape)), g.integers(112, 132, zero.shape)).astype(np.uint8)
            if n == 1:                                      # one element among the zeros: the product below 2^-126 counts
                i, b = np.argwhere(zero)[3]
                blocks[i, b, per - 1], v[s][i, b] = (0x10 if packed else 1), 0
        for C in (v["C"], None):
            _compare(model, v, K, C, (key, (M, N, K), C is None))
