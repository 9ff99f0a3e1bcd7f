"""Sliced FP64 products by themselves: no output is off by more than FP64 arithmetic may be.

The kernel holds a row in fixed point, 62 bits below its largest element.
Every output still has to keep the bound of a chain of FP64 multiply-adds,
element by element of the product's terms: real and imaginary part within
2 K 2^-53 sum_k |a_k||b_k| of the exact value, plus one rounding each for
alpha, the accumulation and the joined result: (2 K + 4) 2^-53.  Rows graded
in opposite directions, disjoint rows, results near and below the smallest
normal number and rows with infinities or NaN are what the fixed point cannot
hold.  The reference is in extended precision (64 bits of mantissa and more).
"""
import ctypes

import numpy as np
import pytest
import torch

from paper_2407_18947_gb300 import _lib

pytestmark = pytest.mark.gpu


class Plan(ctypes.Structure):
    _fields_ = [("swap", ctypes.c_bool), ("nt", ctypes.c_int), ("seg", ctypes.c_int),
                ("nseg", ctypes.c_int), ("spc", ctypes.c_int), ("nsplit", ctypes.c_int),
                ("cost", ctypes.c_double)]


class Operand(ctypes.Structure):
    _fields_ = [("p", ctypes.c_void_p), ("off", ctypes.c_longlong), ("rows", ctypes.c_void_p),
                ("ks", ctypes.c_void_p), ("kc", ctypes.c_bool)]


def _gemm(a, b, alpha, c0, nt, kc, seg=128, spc=1):
    """alpha a b^T (+ c0) for a (M, K), b (N, K); kc: k contiguous in memory."""
    lib = _lib.load()
    f = getattr(lib, "_ZN5rtcc37oz_gemmERKNS_6OzPlanERKNS_9OzOperandES5_iiiP7double2xPKxS9_bdbS7_PixP11CUstream_st")
    i, ll, p, d, bo = ctypes.c_int, ctypes.c_longlong, ctypes.c_void_p, ctypes.c_double, ctypes.c_bool
    f.restype = i
    f.argtypes = [p, p, p, i, i, i, p, ll, p, p, bo, d, bo, p, p, ll, p]
    (M, K), N = a.shape, b.shape[0]
    dev = torch.device("cuda")

    def operand(x):
        t = torch.tensor(x if kc else np.ascontiguousarray(x.T), device=dev)
        r = torch.arange(x.shape[0], device=dev) * (K if kc else 1)
        k = torch.arange(K, device=dev) * (1 if kc else x.shape[0])
        return Operand(t.data_ptr(), 0, r.data_ptr(), k.data_ptr(), kc), (t, r, k)

    A, keep_a = operand(a)
    B, keep_b = operand(b)
    nseg = -(-K // seg)
    plan = Plan(False, nt, seg, nseg, spc, -(-nseg // spc), 0.0)
    C = torch.tensor(np.zeros((M, N), complex) if c0 is None else c0, device=dev)
    cM, cN = torch.arange(M, device=dev) * N, torch.arange(N, device=dev)
    part = torch.empty(plan.nsplit * M * N, dtype=torch.complex128, device=dev)
    err = torch.zeros(1, dtype=torch.int32, device=dev)
    torch.cuda.synchronize()
    f(ctypes.byref(plan), ctypes.byref(A), ctypes.byref(B), M, N, K, C.data_ptr(), 0, cM.data_ptr(),
      cN.data_ptr(), False, alpha, c0 is not None, part.data_ptr(), err.data_ptr(), 0, None)
    torch.cuda.synchronize()
    assert err.item() == 0
    return C.cpu().numpy()


def _check(a, b, alpha=1.0, c0=None, **how):
    c = _gemm(a, b, alpha, c0, **how)
    ar, ai, br, bi = (x.astype(np.longdouble) for x in (a.real, a.imag, b.real, b.imag))
    re, im = ar @ br.T - ai @ bi.T, ar @ bi.T + ai @ br.T
    s = np.hypot(ar, ai) @ np.hypot(br, bi).T * abs(np.longdouble(alpha))
    re, im = re * np.longdouble(alpha), im * np.longdouble(alpha)
    if c0 is not None:
        re, im, s = re + c0.real, im + c0.imag, s + np.abs(c0)
    # one unit of the smallest subnormal number per product and sum
    bound = (2 * a.shape[1] + 4) * (2.0**-53 * s + 5e-324)
    worst = max(np.max((np.abs(c.real - re) / bound)), np.max((np.abs(c.imag - im) / bound)))
    assert worst <= 1.0, float(worst)
    return float(worst)


def _gauss(rng, *shape):
    return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)


HOW = [dict(nt=64, kc=True), dict(nt=48, kc=False), dict(nt=32, kc=True), dict(nt=16, kc=False)]


@pytest.mark.parametrize("how", HOW)
@pytest.mark.parametrize("M,N,K", [(1, 1, 4), (130, 33, 7), (127, 24, 48), (150, 40, 128)])
@pytest.mark.parametrize("spread", [1.0, 1e2, 1e4, 1e8, 1e12, 1e30])
def test_rows_graded_in_opposite_directions(how, M, N, K, spread):
    rng = np.random.default_rng(M + K)
    w = np.logspace(0, np.log10(spread), K)
    _check(_gauss(rng, M, K) * w, _gauss(rng, N, K) / w, **how)
    # every row its own grading, forwards or backwards
    wm = np.where(rng.random((M, 1)) < 0.5, w, w[::-1])
    wn = np.where(rng.random((N, 1)) < 0.5, w, w[::-1])
    _check(_gauss(rng, M, K) * wm, _gauss(rng, N, K) * wn, **how)


@pytest.mark.parametrize("how", HOW)
def test_segments_alpha_and_accumulation(how):
    rng = np.random.default_rng(5)
    for K, seg, spc in ((300, 128, 1), (300, 128, 3), (700, 64, 4)):
        w = np.logspace(0, 9, K)
        a, b = _gauss(rng, 140, K) * w, _gauss(rng, 20, K) / w
        for alpha, c0 in ((1.0, None), (-0.25, _gauss(rng, 140, 20)), (0.7, _gauss(rng, 140, 20) * 1e3)):
            _check(a, b, alpha, c0, seg=seg, spc=spc, **how)


@pytest.mark.parametrize("how", HOW)
def test_sparse_and_disjoint_rows(how):
    rng = np.random.default_rng(6)
    M, N, K = 140, 35, 64
    a, b = _gauss(rng, M, K), _gauss(rng, N, K)
    a[:, ::2] *= 1e-25            # the large elements never meet
    b[:, 1::2] *= 1e-25
    a[3], b[4] = 0.0, 0.0
    a[5, 1:], b[6, :-1] = 0.0, 0.0
    _check(a, b, **how)
    a, b = a.real + 0j, b.real + 0j   # purely real operands
    _check(a, b, **how)
    c = _gemm(a, 1j * b, 1.0, None, **how)
    assert (c.real == 0.0).all()


@pytest.mark.parametrize("how", HOW)
@pytest.mark.parametrize("ea,eb", [(-160, -150), (-307, 0), (-320, 290), (-323, 300), (150, 150), (-300, -300)])
def test_near_the_ends_of_the_range(how, ea, eb):
    rng = np.random.default_rng(7)
    a, b = _gauss(rng, 130, 40), _gauss(rng, 20, 40)
    a, b = a * 10.0**(ea + 20) * 1e-20, b * 10.0**(eb - 20) * 1e20
    _check(a, b, **how)


@pytest.mark.parametrize("how", HOW)
def test_digits_all_of_the_largest_size(how):
    """Equal elements whose digits are all 127 (or -128): the sums of digit
    products beyond 2^24 are not exact any more."""
    for word in (0x3F7F7F7F7F7F7F7F, 0x3E7F7F7F7F7F7F80, 0x2080808080808080):
        x = float(word >> 10) * 2.0**-52
        a, b = np.full((130, 128), x * (1 + 1j)), np.full((20, 128), x * (1 - 1j))
        a[1] *= 0.5
        _check(a, b, **how)


@pytest.mark.parametrize("how", HOW)
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_non_finite_elements_reach_their_outputs_only(how, bad):
    rng = np.random.default_rng(8)
    a, b = _gauss(rng, 130, 40), _gauss(rng, 20, 40)
    a[7, 11] = bad
    b[3, 5] = complex(0.0, bad)
    b[4] = 0.0                        # 0 x inf and 0 x nan are NaN
    c = _gemm(a, b, 1.0, None, **how)
    ok = np.isfinite(c.view(float)).reshape(130, 20, 2).all(-1)
    want = np.ones((130, 20), bool)
    want[7], want[:, 3] = False, False
    assert (ok == want).all()
