"""The products on 16-bit slices by themselves (dla.cuh), entry by entry: each
row of A and column of B has its own scale, so every entry is held against the
largest entries, or the norms, of its own row and column.

Tolerances: FP64 in seven digits, K 2^-54 (both operands' rounding) + K 2^-59
(digit products left out) times the row's and the column's largest entries, and
2^-53 of the entry (rounded once, and once more per part of a split K).  FP32
arithmetic: two FP16 slices of each operand drop 2^-22 of a product, FP32 sums over
a chunk of K a few 2^-24 more: 2^-20 of the row's and the column's norms.
"""

import ctypes
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

F64, F32, BF16, F16 = 0, 1, 2, 3  # bsrht::DT


class _Arena(ctypes.Structure):  # bsrht::Arena
    _fields_ = [("base", ctypes.c_void_p), ("cap", ctypes.c_size_t), ("used", ctypes.c_size_t),
                ("high", ctypes.c_size_t), ("measure", ctypes.c_bool), ("lean", ctypes.c_bool)]


class _Dla(ctypes.Structure):  # bsrht::Dla
    _fields_ = [("s", ctypes.c_void_p), ("status", ctypes.c_void_p)]


class _Products:
    """The library's internal products, by their mangled names."""

    def __init__(self, lib):
        i64, vp, ci, cb = ctypes.c_int64, ctypes.c_void_p, ctypes.c_int, ctypes.c_bool
        head = [ctypes.POINTER(_Dla), ctypes.POINTER(_Arena)]
        self.int8x7 = getattr(lib, "_ZN5bsrht11gemm_int8x7ERKNS_3DlaERNS_5ArenaElllPKdlbS6_lPdlbb")
        self.int8x7.argtypes = head + [i64, i64, i64, vp, i64, cb, vp, i64, vp, i64, cb, cb]
        self.f32x2 = getattr(lib, "_ZN5bsrht10gemm_f32x2ERKNS_3DlaERNS_5ArenaElllPKflNS_2DTEPKvlS7_PvlbPf")
        self.f32x2.argtypes = head + [i64, i64, i64, vp, i64, ci, vp, i64, ci, vp, i64, cb, vp]
        self.a16 = getattr(lib, "_ZN5bsrht8gemm_a16ERKNS_3DlaERNS_5ArenaENS_2DTElllPKvlS5_S7_lPflS8_")
        self.a16.argtypes = head + [ci, i64, i64, i64, vp, i64, ci, vp, i64, vp, i64, vp]
        self.signs = getattr(lib, "_ZN5bsrht14sign_normalizeERKNS_3DlaERNS_5ArenaEPdllS5_l")
        self.signs.argtypes = head + [vp, i64, i64, vp, i64]
        self.scratch = torch.empty(1 << 30, device="cuda", dtype=torch.uint8)
        self.status = torch.zeros(64, device="cuda", dtype=torch.int32)

    def measure(self, fn, *args):
        """Bytes of scratch that a call of these sizes takes, with the slack that the workspace queries add."""
        d = _Dla(None, None)
        ar = _Arena(None, 0, 0, 0, True, False)
        assert fn(ctypes.byref(d), ctypes.byref(ar), *args) == 0
        return ar.high + 256

    def run(self, fn, *args, scratch=None):
        torch.cuda.synchronize()
        d = _Dla(torch.cuda.current_stream().cuda_stream, self.status.data_ptr())
        ar = _Arena(self.scratch.data_ptr(), scratch or self.scratch.numel(), 0, 0, False, False)
        st = fn(ctypes.byref(d), ctypes.byref(ar), *args)
        torch.cuda.synchronize()
        assert st == 0 and int(self.status[0]) == 0


@pytest.fixture(scope="module")
def prod():
    import paper_2210_11295_gb300._binding as b

    return _Products(b.lib)


def _spread(rng, rows, cols, axis, lo, hi):
    x = rng.standard_normal((rows, cols))
    return x * np.exp2(rng.integers(lo, hi + 1, size=(rows, 1) if axis == 0 else (1, cols)))


@pytest.mark.parametrize("K", [1, 40, 1000])
def test_digits_of_one_sign(prod, K):
    """Every digit product that is left out has the same sign."""
    t = 65 * 2**48 - 128 * ((2**48 - 1) // 255)  # digits 65, -128, -128, ...
    v = float(t)
    assert int(v) == t
    M, N = 130, 70
    a = torch.full((M, K), v, device="cuda", dtype=torch.float64)
    b = torch.full((K, N), v, device="cuda", dtype=torch.float64)
    c = torch.empty(M, N, device="cuda", dtype=torch.float64)
    prod.run(prod.int8x7, M, N, K, a.data_ptr(), K, False, b.data_ptr(), N, c.data_ptr(), N, False, False)
    exact = Fraction(t) ** 2 * K
    got = c.unique().cpu().tolist()
    assert len(got) == 1
    assert abs(Fraction(got[0]) - exact) <= exact * (Fraction(1, 2**53) + Fraction(1, 2**59))


@pytest.mark.parametrize("M,N,K,trans,gram,upper", [
    (129, 65, 257, False, False, False),
    (300, 300, 300, False, False, True),
    (100, 70, 1000, True, False, False),
    (130, 130, 4000, True, True, False),
])
def test_fp64_per_entry(prod, M, N, K, trans, gram, upper):
    rng = np.random.default_rng(M + K)
    a = _spread(rng, M, K, 0, -30, 30)  # op(A)
    b = a.T.copy() if gram else _spread(rng, K, N, 1, -30, 30)
    if upper:
        b = np.triu(b)
    stored = torch.from_numpy(np.ascontiguousarray(a.T if trans else a)).cuda()
    bd = stored if gram else torch.from_numpy(b).cuda()
    c = torch.empty(M, N, device="cuda", dtype=torch.float64)
    prod.run(prod.int8x7, M, N, K, stored.data_ptr(), M if trans else K, trans, bd.data_ptr(), N, c.data_ptr(), N,
             upper, gram)
    exact = np.matmul(a.astype(np.longdouble), b.astype(np.longdouble))
    largest = np.abs(a).max(1)[:, None] * np.abs(b).max(0)[None, :]
    off = np.abs(c.cpu().numpy() - exact)
    parts = 64  # a split K: sums of at most as many rounded parts
    assert np.all(off <= (K * 2.0**-54 + K * 2.0**-59) * largest + 2.0**-53 * np.abs(exact)
                  + (0 if K < 512 else parts * 2.0**-53 * K * largest))


def _check_fp32(c, a, b):
    exact = a @ b
    norms = np.linalg.norm(a, axis=1)[:, None] * np.linalg.norm(b, axis=0)[None, :]
    assert np.all(np.abs(c.double().cpu().numpy() - exact) <= 2.0**-20 * norms)


def _f32x2(prod, a, b, f64out=False):
    (M, K), N = a.shape, b.shape[1]
    lda = (K + 3) // 4 * 4
    buf = torch.zeros(M, lda)
    buf[:, :K] = torch.from_numpy(a)
    ad, bd = buf.cuda(), torch.from_numpy(b).cuda()
    c = torch.empty(M, N, device="cuda", dtype=torch.float64 if f64out else torch.float32)
    prod.run(prod.f32x2, M, N, K, ad.data_ptr(), lda, F64, bd.data_ptr(), N, F64 if f64out else F32, c.data_ptr(), N,
             False, None)
    return c


def _a16(prod, a, b):
    (M, K), N = a.shape, b.shape[1]
    ad, bd = a.cuda(), torch.from_numpy(b).cuda()
    c = torch.empty(M, N, device="cuda", dtype=torch.float32)
    ct = torch.empty(N, M, device="cuda", dtype=torch.float32)
    prod.run(prod.a16, BF16 if a.dtype is torch.bfloat16 else F16, M, N, K, ad.data_ptr(), K, F64, bd.data_ptr(), N,
             c.data_ptr(), N, ct.data_ptr())
    assert torch.allclose(ct.T, c, rtol=0, atol=0, equal_nan=True)
    return c


@pytest.mark.parametrize("M,N,K,f64out", [(300, 130, 257, False), (257, 272, 1000, True), (12290, 40, 96, False)])
def test_fp32_per_row(prod, M, N, K, f64out):
    rng = np.random.default_rng(M + K)
    a = _spread(rng, M, K, 0, -40, 0).astype(np.float32)
    b = _spread(rng, K, N, 1, -20, 20)
    _check_fp32(_f32x2(prod, a, b, f64out), a.astype(np.float64), b)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float16])
@pytest.mark.parametrize("M,N,K", [(300, 130, 256), (257, 272, 1000)])
def test_16bit_per_row(prod, dtype, M, N, K):
    rng = np.random.default_rng(M + K)
    a = torch.from_numpy(_spread(rng, M, K, 0, -10, 0)).to(dtype)
    b = _spread(rng, K, N, 1, -20, 20)
    _check_fp32(_a16(prod, a, b), a.double().numpy(), b)


@pytest.mark.parametrize("ea,eb", [(118, -4), (105, 10), (-110, 4), (60, -100), (-60, 100)])
def test_ends_of_the_range(prod, ea, eb):
    """FP32 and BF16 data near the ends of FP32's range, products within it."""
    rng = np.random.default_rng(7)
    a = rng.standard_normal((300, 128)) * 2.0**ea
    b = rng.standard_normal((128, 40)) * 2.0**eb
    a32, b32 = a.astype(np.float32), b.astype(np.float32).astype(np.float64)
    _check_fp32(_f32x2(prod, a32, b32), a32.astype(np.float64), b32)
    a16 = torch.from_numpy(a).to(torch.bfloat16)
    _check_fp32(_a16(prod, a16, b32), a16.double().numpy(), b32)


@pytest.mark.parametrize("M,N,K,trans,gram", [
    (1000, 130, 257, False, False),   # split K
    (40000, 100, 700, False, False),  # several passes over the rows
    (300, 200, 60000, True, False),   # several passes over K
    (256, 256, 100000, True, True),
])
def test_fp64_scratch_as_measured(prod, M, N, K, trans, gram):
    """The scratch that is measured for a product holds it: the same launches as with ample scratch."""
    import paper_2210_11295_gb300 as lib

    a = torch.randn((K, M) if trans else (M, K), device="cuda", dtype=torch.float64)
    b = a if gram else torch.randn(K, N, device="cuda", dtype=torch.float64)
    c = torch.empty(M, N, device="cuda", dtype=torch.float64)
    args = (M, N, K, a.data_ptr(), M if trans else K, trans, b.data_ptr(), N, c.data_ptr(), N, False, gram)

    def launches(scratch):
        before = lib.bsrht_kernel_launches()
        prod.run(prod.int8x7, *args, scratch=scratch)
        return lib.bsrht_kernel_launches() - before

    ample = launches(None)
    full = c.clone()
    assert launches(prod.measure(prod.int8x7, *args)) == ample
    assert torch.equal(c, full)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_nonfinite_stays_in_its_row_or_column(prod, bad):
    rng = np.random.default_rng(3)
    M, N, K = 300, 130, 256
    a, b = rng.standard_normal((M, K)), rng.standard_normal((K, N))
    rows, cols = np.arange(M) == 77, np.arange(N) == 5
    touched = rows[:, None] | cols[None, :]
    an, bn = a.copy(), b.copy()
    an[77, 3], bn[9, 5] = bad, bad
    ad, bd = torch.from_numpy(an).cuda(), torch.from_numpy(bn).cuda()
    c = torch.empty(M, N, device="cuda", dtype=torch.float64)
    prod.run(prod.int8x7, M, N, K, ad.data_ptr(), K, False, bd.data_ptr(), N, c.data_ptr(), N, False, False)
    got = c.cpu().numpy()
    assert np.all(np.isnan(got[touched]))
    assert np.all(np.abs(got - a @ b)[~touched] <= 1e-12)
    a16 = torch.from_numpy(an).to(torch.bfloat16)
    for c, vals in ((_f32x2(prod, an.astype(np.float32), bn), a), (_a16(prod, a16, bn), a16.double().numpy())):
        got = c.double().cpu().numpy()
        assert not np.any(np.isfinite(got[touched]))
        clean = np.where(np.isfinite(vals), vals, 0.0)
        norms = np.linalg.norm(clean, axis=1)[:, None] * np.linalg.norm(b, axis=0)[None, :]
        assert np.all(np.abs(got - clean @ b)[~touched] <= (2.0**-20 * norms)[~touched])


@pytest.mark.parametrize("n,k", [(1, 1), (5000, 7), (70000, 100), (300, 300), (4097, 1)])
def test_signs_with_ties(prod, n, k):
    """The sign of a column is that of its first largest entry."""
    rng = np.random.default_rng(n + k)
    u = rng.integers(-2, 3, size=(n, k)).astype(np.float64)  # many entries tie for the largest
    v = rng.standard_normal((9, k))
    ud, vd = torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda()
    prod.run(prod.signs, ud.data_ptr(), n, k, vd.data_ptr(), 9)
    sign = np.where(u[np.argmax(np.abs(u), axis=0), np.arange(k)] < 0, -1.0, 1.0)
    assert np.array_equal(ud.cpu().numpy(), u * sign)
    assert np.array_equal(vd.cpu().numpy(), v * sign)
