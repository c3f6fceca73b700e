"""Rows off the 16-byte grid: K of any length, in every element type, on the tiled kernels, and
operands at any byte; against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2608_12114_gb300 import build, synth, wt

pytestmark = pytest.mark.gpu
F32, BF16, F16, I8 = wt.WT_F32, wt.WT_BF16, wt.WT_F16, wt.WT_I8
ES = {F32: 4, BF16: 2, F16: 2, I8: 1}

# (M, bytes of a row, bytes past a 16-byte boundary of W and of x): matrices and rows smaller
# than a vector; rows of one phase that fill 16 and 32 lanes and of another that need one more;
# every row count of a stage; 8 rows and fewer; the longest unsegmented row (504 vectors; int8:
# 184) and the first segmented one; a partial last segment; aligned rows at unaligned addresses
SHAPES = [(1, 4, 0, 0), (5, 4, 4, 4), (3, 20, 0, 0), (1000, 12, 8, 0), (33, 232, 4, 8), (33, 244, 0, 4), (40, 256, 4, 0),
          (70, 496, 12, 0), (70, 508, 4, 0), (90, 516, 4, 0), (65, 1012, 0, 0), (65, 1028, 8, 0), (300, 2940, 0, 0),
          (300, 2948, 4, 4), (41, 4084, 0, 0), (41, 4100, 0, 0), (129, 5460, 0, 0), (7, 6132, 0, 0), (50, 8060, 4, 0),
          (50, 8064, 4, 0), (50, 8068, 0, 0), (37, 8192, 0, 8), (37, 8196, 4, 0), (19, 12300, 0, 0), (9, 32636, 0, 0),
          (5, 65540, 4, 0), (3, 131076, 0, 12)]


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available()
    build.build()
    wt.lib()
    return torch


def weights(rng, dtype, n):
    if dtype == I8:
        return rng.integers(-128, 128, n).astype(np.int8).view(np.uint8)
    v = rng.standard_normal(n).astype(np.float32)
    return synth.f32_to_bf16_bits(v).view(np.uint8) if dtype == BF16 else \
        v.astype(np.float16 if dtype == F16 else np.float32).view(np.uint8)


def at(torch, data, off):
    """`data` on the device, `off` bytes past a 16-byte boundary, among bytes of 0xff (NaN in
    every float type: a value read past an operand shows)."""
    buf = torch.full((data.size + 64,), 255, dtype=torch.uint8, device="cuda")
    buf[16 + off:16 + off + data.size] = torch.from_numpy(np.ascontiguousarray(data)).cuda()
    return buf, buf.data_ptr() + 16 + off


def bound(K):
    """|fp32 sum of K products - exact| <= K u sum|w x|, and the row scale's rounding."""
    return (K + 4) * 2.0 ** -24


@pytest.mark.parametrize("dtype", [F32, BF16, F16, I8])
@pytest.mark.parametrize("odd", [0, 1])
def test_ragged_rows_against_oracle(torch, dtype, odd):
    """Every shape in one pass with an aligned matrix, then alone (the same bits).  odd: one
    element fewer per row, so that rows of 1- and 2-byte types start at every phase."""
    rng = np.random.default_rng(100 * dtype + odd)
    es = ES[dtype]
    shapes = [(M, max(1, kb // es - odd), wo - wo % es, xo - xo % (2 if dtype == I8 else es))
              for M, kb, wo, xo in SHAPES] + [(64, 1024, 0, 0)]
    cs = []
    for M, K, wo, xo in shapes:
        W, x = weights(rng, dtype, M * K), weights(rng, F16 if dtype == I8 else dtype, K)
        s = rng.uniform(0.001, 0.02, M).astype(np.float16).view(np.uint8) if dtype == I8 else None
        wb, wp = at(torch, W, wo)
        xb, xp = at(torch, x, xo)
        sb, sp = at(torch, s, 0) if s is not None else (None, 0)
        y = torch.full((M,), float("nan"), dtype=torch.float32, device="cuda")
        ref = oracle.gemv_q8(W, s, M, K, x) if dtype == I8 else oracle.gemv(W, dtype, M, K, x)
        cs.append((M, K, wp, xp, sp, y, ref, (wb, xb, sb)))
    with wt.Handle([]) as h:
        h.pass_([wt.gemv_desc(wp, dtype, M, K, xp, y.data_ptr(), scale=sp) for M, K, wp, xp, sp, y, _, _ in cs], 0)
        torch.cuda.synchronize()
        assert h.device_status() == 0
        for M, K, wp, xp, sp, y, (yhat, a), _ in cs:
            err = oracle.gemv_error(y.cpu().numpy(), yhat, a)
            assert err <= bound(K), (dtype, M, K, err)
        for M, K, wp, xp, sp, y, _, _ in cs:
            y2 = torch.full_like(y, float("nan"))
            h.pass_([wt.gemv_desc(wp, dtype, M, K, xp, y2.data_ptr(), scale=sp)], 0)
            assert torch.equal(y2, y), (dtype, M, K)
        assert h.device_status() == 0


# (M, bytes of a row, bytes past a 16-byte boundary of W and of X): a 16-row tile and a 64-row
# super block and one more row; one 4-vector group; 84 vectors (one chunk) and one more; several
# uneven chunks; aligned rows, also at unaligned addresses; on both sides of the longest short
# rows (1024 bytes; int8: 512); several stages of 32-row groups
COL_SHAPES = [(1, 4, 0, 0), (17, 20, 4, 4), (64, 64, 4, 0), (65, 132, 0, 0), (33, 1340, 0, 4), (16, 1344, 4, 0),
              (80, 1348, 0, 0), (130, 2732, 8, 8), (40, 5460, 0, 0), (23, 20004, 4, 4), (1100, 32, 0, 0), (600, 48, 0, 0),
              (70, 1024, 0, 0), (33, 1028, 4, 0), (200, 2048, 0, 0), (35, 2052, 0, 0), (100, 300, 0, 2), (70, 508, 2, 0),
              (100, 512, 4, 0), (70, 514, 0, 0), (70, 516, 2, 2), (70, 1022, 0, 0), (100, 1024, 2, 0), (70, 1026, 0, 0)]


@pytest.mark.parametrize("dtype", [BF16, F16, I8])
@pytest.mark.parametrize("T", [1, 8, 9, 16])
def test_ragged_columns_against_oracle(torch, dtype, T):
    """As above with T activation columns.  The tensor cores truncate where fp32 additions
    round, so each of a sum's K additions may lose twice as much."""
    rng = np.random.default_rng(1000 * dtype + T)
    es = ES[dtype]
    cs = []
    for odd in (0, 1):
        for M, kb, wo, xo in COL_SHAPES:
            K = max(1, kb // es - odd)
            W, X = weights(rng, dtype, M * K), weights(rng, F16 if dtype == I8 else dtype, T * K)
            s = rng.uniform(0.001, 0.02, M).astype(np.float16).view(np.uint8) if dtype == I8 else None
            wb, wp = at(torch, W, wo - wo % es)
            xb, xp = at(torch, X, xo)
            sb, sp = at(torch, s, 0) if s is not None else (None, 0)
            y = torch.full((T * M,), float("nan"), dtype=torch.float32, device="cuda")
            cs.append((M, K, wp, xp, sp, y, oracle.gemv_cols(W, dtype, M, K, X, T, scale=s), (wb, xb, sb)))
    with wt.Handle([]) as h:
        h.pass_([wt.gemv_desc(wp, dtype, M, K, xp, y.data_ptr(), scale=sp, cols=T) for M, K, wp, xp, sp, y, _, _ in cs], 0)
        torch.cuda.synchronize()
        assert h.device_status() == 0
        for M, K, wp, xp, sp, y, (yhat, a), _ in cs:
            err = oracle.gemv_error(y.cpu().numpy(), yhat.reshape(-1), a.reshape(-1))
            assert err <= 2 * bound(K), (dtype, M, K, T, err)
        for M, K, wp, xp, sp, y, _, _ in cs:
            y2 = torch.full_like(y, float("nan"))
            h.pass_([wt.gemv_desc(wp, dtype, M, K, xp, y2.data_ptr(), scale=sp, cols=T)], 0)
            assert torch.equal(y2, y), (dtype, M, K, T)
        assert h.device_status() == 0


@pytest.mark.parametrize("dtype", [F32, BF16, F16, I8])
@pytest.mark.parametrize("T", [0, 3, 16])
def test_operands_off_their_element_size(torch, dtype, T):
    """W and x at any byte, elements across the boundaries of every load: short rows, whole rows
    and rows long enough for column segments, one column and several (no f32)."""
    if T and dtype == F32:
        pytest.skip("f32 weights have one column")
    rng = np.random.default_rng(17 * dtype + T)
    es = ES[dtype]
    cs = []
    for wo, xo in ((1, 0), (2, 1), (3, 3), (15, 0), (0, 1), (16, 7)):
        for M, kb in ((9, 20), (33, 256), (70, 1028), (50, 2732), (21, 8064), (19, 12300)):
            K = kb // es
            W, X = weights(rng, dtype, M * K), weights(rng, F16 if dtype == I8 else dtype, max(1, T) * K)
            s = rng.uniform(0.001, 0.02, M).astype(np.float16).view(np.uint8) if dtype == I8 else None
            wb, wp = at(torch, W, wo)
            xb, xp = at(torch, X, xo)
            sb, sp = at(torch, s, 0) if s is not None else (None, 0)
            y = torch.full((max(1, T) * M,), float("nan"), dtype=torch.float32, device="cuda")
            ref = oracle.gemv_cols(W, dtype, M, K, X, T, scale=s) if T else \
                oracle.gemv_q8(W, s, M, K, X) if dtype == I8 else oracle.gemv(W, dtype, M, K, X)
            cs.append((wt.gemv_desc(wp, dtype, M, K, xp, y.data_ptr(), scale=sp, cols=T), M, K, wo, xo, y, ref, (wb, xb, sb)))
    with wt.Handle([]) as h:
        h.pass_([c[0] for c in cs], 0)
        torch.cuda.synchronize()
        assert h.device_status() == 0
    for _, M, K, wo, xo, y, (yhat, a), _ in cs:
        err = oracle.gemv_error(y.cpu().numpy(), yhat.reshape(-1), a.reshape(-1))
        assert err <= (2 if T else 1) * bound(K), (dtype, M, K, T, wo, xo, err)


def floats(dtype, raw):
    if dtype == F16:
        return raw.view(np.float16).astype(np.float32)
    return (raw.view(np.uint16).astype(np.uint32) << 16).view(np.float32)


def fma_chains(W, X):
    """W X[t] in fp32 as one warp per row sums it: a chain of FMAs per lane over every 32nd
    product, then the lanes in a tree.  (A product of these types is exact in 64 bits.)"""
    T, (M, K) = X.shape[0], W.shape
    acc = np.zeros((T, M, 32), np.float32)
    for k in range(0, K, 32):
        w, x = W[:, k:k + 32].astype(np.float64), X[:, k:k + 32].astype(np.float64)
        n = w.shape[1]
        acc[:, :, :n] = (w[None] * x[:, None] + acc[:, :, :n]).astype(np.float32)
    while acc.shape[2] > 1:
        h = acc.shape[2] // 2
        acc = acc[:, :, :h] + acc[:, :, h:]
    return acc[:, :, 0]


@pytest.mark.parametrize("dtype", [BF16, F16, I8])
@pytest.mark.parametrize("T", [3, 8, 12])
def test_ragged_columns_are_as_exact_as_fp32_fmas(torch, dtype, T):
    """The 2-norm error against 64-bit sums is no larger than that of fp32 FMAs, which these calls
    had before the tensor cores: rows on both sides of the short-row limit and of the lines from
    which one MMA per step is enough.  6144 and more outputs put the sampling error of a ratio at
    about 2 %."""
    rng = np.random.default_rng(31 * dtype + T)
    M = 2048
    with wt.Handle([]) as h:
        for K in (33, 77, 200 + (dtype != I8), 333, 511, 513, 777, 1027, 2049 if dtype == I8 else 1153, 2731):
            W, X = weights(rng, dtype, M * K), weights(rng, F16 if dtype == I8 else dtype, T * K)
            s = np.ones(M, np.float16).view(np.uint8)
            wb, wp = at(torch, W, 0 if K % 8 else 2)
            xb, xp = at(torch, X, 0)
            sb, sp = at(torch, s, 0)
            y = torch.full((T * M,), float("nan"), dtype=torch.float32, device="cuda")
            h.pass_([wt.gemv_desc(wp, dtype, M, K, xp, y.data_ptr(), scale=sp if dtype == I8 else 0, cols=T)], 0)
            Wf = W.view(np.int8).astype(np.float32) if dtype == I8 else floats(dtype, W)
            Wf, Xf = Wf.reshape(M, K), floats(F16 if dtype == I8 else dtype, X).reshape(T, K)
            exact = Xf.astype(np.float64) @ Wf.astype(np.float64).T
            ours = np.linalg.norm(y.cpu().numpy().reshape(T, M) - exact)
            theirs = np.linalg.norm(fma_chains(Wf, Xf) - exact)
            assert ours <= 1.02 * theirs, (dtype, T, K, ours / theirs)
        assert h.device_status() == 0


@pytest.mark.parametrize("dtype", [BF16, F16, I8])
@pytest.mark.parametrize("T", [5, 16])
def test_short_rows_over_many_stages(torch, dtype, T):
    """Short rows, aligned and ragged, with some 200 KB for each CTA: the ring of five 32 KB stages
    wraps within one matrix.  Against 64-bit sums, Y NaN-filled first."""
    g = torch.Generator("cuda").manual_seed(50 + T)
    tdt = {BF16: torch.bfloat16, F16: torch.float16, I8: torch.int8}[dtype]
    shapes = ((60001, 509), (30001 * 20, 48)) if dtype == I8 else ((30001, 512), (30001, 511), (40 * 30001, 13))
    with wt.Handle([]) as h:
        for M, K in shapes:
            if dtype == I8:
                W = torch.randint(-128, 128, (M, K), dtype=tdt, device="cuda", generator=g)
                s = torch.rand(M, device="cuda", generator=g).half()
            else:
                W, s = torch.empty(M, K, dtype=tdt, device="cuda").normal_(0, 0.02, generator=g), None
            X = torch.empty(T, K, dtype=torch.float16 if dtype == I8 else tdt, device="cuda").normal_(0, 1, generator=g)
            y = torch.full((T * M,), float("nan"), device="cuda")
            h.pass_([wt.gemv_desc(W.data_ptr(), dtype, M, K, X.data_ptr(), y.data_ptr(), cols=T,
                                  scale=s.data_ptr() if s is not None else 0)], 0)
            ref, mag = X.double() @ W.double().t(), X.double().abs() @ W.double().abs().t()
            if s is not None:
                ref, mag = ref * s.double(), mag * s.double()
            assert ((y.view(T, M).double() - ref).abs() <= 2 * bound(K) * mag).all(), (dtype, T, M, K)
        assert h.device_status() == 0


@pytest.mark.parametrize("T", [0, 8, 12])
def test_small_int8_launches_stay_exact(torch, T):
    """Launches of fewer than 304 blocks of 128 rows, evenly dealt ones among them: the tensor
    cores truncate, so a sum of them may lose twice what fp32 FMAs lose, and no more."""
    rng = np.random.default_rng(77 + T)
    with wt.Handle([]) as h:
        for M, K in ((8192, 128), (8192, 256), (8192, 512), (4096, 576), (2048, 1024)):
            W, X = weights(rng, I8, M * K), weights(rng, F16, max(1, T) * K)
            wb, wp = at(torch, W, 0)
            xb, xp = at(torch, X, 0)
            sb, sp = at(torch, np.ones(M, np.float16).view(np.uint8), 0)
            y = torch.full((max(1, T) * M,), float("nan"), dtype=torch.float32, device="cuda")
            h.pass_([wt.gemv_desc(wp, I8, M, K, xp, y.data_ptr(), scale=sp, cols=T)], 0)
            Wf, Xf = W.view(np.int8).astype(np.float32).reshape(M, K), floats(F16, X).reshape(-1, K)
            exact = Xf.astype(np.float64) @ Wf.astype(np.float64).T
            ours = np.linalg.norm(y.cpu().numpy().reshape(-1, M) - exact)
            theirs = np.linalg.norm(fma_chains(Wf, Xf) - exact)
            assert ours <= 2 * theirs, (T, M, K, ours / theirs)
        assert h.device_status() == 0


@pytest.mark.parametrize("K", [45, 1031])
def test_ragged_columns_with_infinities_and_overflow(torch, K):
    """An infinite weight, sums that leave fp32 on either side, and a NaN, in rows of their own:
    y as IEEE sums give it, and the other rows untouched."""
    T, M = 5, 40
    W = torch.full((M, K), 0.5, dtype=torch.bfloat16, device="cuda")
    W[3, 7] = float("inf")
    W[4, K - 1] = float("-inf")
    W[17, :] = 3e38
    W[18, :] = -3e38
    W[33, 0] = float("nan")
    X = torch.full((T, K), 1.0, dtype=torch.bfloat16, device="cuda")
    y = torch.full((T * M,), float("nan"), device="cuda")
    with wt.Handle([]) as h:
        h.pass_([wt.gemv_desc(W.data_ptr(), BF16, M, K, X.data_ptr(), y.data_ptr(), cols=T)], 0)
        torch.cuda.synchronize()
        assert h.device_status() == 0
    y = y.view(T, M).cpu()
    inf = float("inf")
    for r in range(M):
        want = {3: inf, 4: -inf, 17: inf, 18: -inf}.get(r, 0.5 * K)
        assert (torch.isnan(y[:, r]) if r == 33 else y[:, r] == want).all(), (r, y[:, r])
