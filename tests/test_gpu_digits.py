"""The FP64 Grams and products formed from 8-bit digits (csrc/oz.cu), against
exact sums, called by their C++ names.

The bound of a sum of K products a b, each block's entries held against the
largest magnitude of its column: both entries are cut at 2^-62 of it, and of the 64 digit products 36 are kept.
The dropped ones are at most sum_{d >= 8} (15 - d) 2^14 2^(8 (14 - d)) = 2^64.9
of the 2^124 that the largest entries' product has, 2^-59.1 of it, the cuts
2 2^-63: together below 2^-58.9 K 2^ea 2^eb, whatever the entries, with 2^e the
power of two above the column's largest magnitude. On top come
the roundings of the result: two per slice of rows and one per slice added."""
import ctypes as ct

import numpy as np
import pytest

import trm_inputs as ti
from oracle import trm as otrm

from . import gpu_util as gu

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


class _Block(ct.Structure):
    _fields_ = [("digits", ct.c_void_p), ("scale", ct.c_void_p),
                ("N", ct.c_int64), ("m", ct.c_int)]


class _Small(ct.Structure):
    _fields_ = [("digits", ct.c_void_p), ("scale", ct.c_void_p)]


class _Digits:
    """oz_slice, oz_gram and oz_mult on numpy blocks."""

    def __init__(self, path):
        self.lib = ct.CDLL(path)

    def _size(self, name, a, b):
        f = getattr(self.lib, name)
        f.restype = ct.c_size_t
        return f(a, b)

    def slice(self, A):
        import torch
        N, m = A.shape
        src = gu.to_dev(A)
        mem = torch.zeros(self._size("_ZN3trm14oz_block_bytesEli",
                                     ct.c_int64(N), m),
                          dtype=torch.uint8, device="cuda")
        scale = gu.to_dev(np.zeros(m))
        b = _Block(mem.data_ptr(), scale.data_ptr(), 0, 0)
        self.lib._ZN3trm8oz_sliceEliPKdlRNS_7OzBlockEP11CUstream_stS1_PKNS_11IterScalarsEdd(
            ct.c_int64(N), m, ct.c_void_p(src.data_ptr()), ct.c_int64(N),
            ct.byref(b), ct.c_void_p(gu.stream()), None, None,
            ct.c_double(1.0), ct.c_double(0.0))
        torch.cuda.synchronize()
        return b, (mem, scale)

    def gram(self, A, B):
        import torch
        a, keep_a = self.slice(A)
        b, keep_b = self.slice(B)
        m, n = A.shape[1], B.shape[1]
        out = gu.empty(m, n, np.float64)
        cap = 160 * m * n
        part, err = gu.to_dev(np.zeros(cap)), gu.to_dev(np.zeros(4, np.int32))
        self.lib._ZN3trm7oz_gramEPKNS_7OzBlockEiRS1_PdS4_mPiP11CUstream_st(
            ct.byref(a), 1, ct.byref(b), ct.c_void_p(out.data_ptr()),
            ct.c_void_p(part.data_ptr()), ct.c_size_t(cap),
            ct.c_void_p(err.data_ptr()), ct.c_void_p(gu.stream()))
        torch.cuda.synchronize()
        assert int(err[0]) == 0
        return gu.from_dev(out)

    def mult(self, A, M, tri=False):
        import torch
        a, keep = self.slice(A)
        N, k = A.shape
        n = M.shape[1]
        Md, Y = gu.to_dev(M), gu.empty(N, n, np.float64)
        mem = torch.zeros(self._size("_ZN3trm14oz_small_bytesEii", k, n),
                          dtype=torch.uint8, device="cuda")
        scale, err = gu.to_dev(np.zeros(n)), gu.to_dev(np.zeros(4, np.int32))
        w = _Small(mem.data_ptr(), scale.data_ptr())
        self.lib._ZN3trm7oz_multERKNS_7OzBlockEiPKdbRKNS_7OzSmallEPdlPiP11CUstream_stPKi(
            ct.byref(a), n, ct.c_void_p(Md.data_ptr()), ct.c_bool(tri),
            ct.byref(w), ct.c_void_p(Y.data_ptr()), ct.c_int64(N),
            ct.c_void_p(err.data_ptr()), ct.c_void_p(gu.stream()), None)
        torch.cuda.synchronize()
        assert int(err[0]) == 0
        return gu.from_dev(Y)


@pytest.fixture(scope="module")
def digits():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1108_4509_gb300 as trm
    return _Digits(trm.LIB_PATH)


def _extreme(shape, rng, last):
    """Doubles in (-1, -1/2] whose balanced digits are -63, five of -128..-125,
    `last` = an even one of these, 0: all signs equal, every digit near its end.
    Returns them with their digits."""
    d = rng.integers(-128, -124, size=(8,) + shape)
    d[0], d[6], d[7] = -63, last, 0
    q = sum(d[k].astype(object) << (8 * (7 - k)) for k in range(8))
    x = np.array([[float(v) for v in row] for row in q])
    assert all(int(x[i, j]) == q[i, j] for i in range(2) for j in range(2))
    return np.asfortranarray(x * 2.0 ** -62), d.astype(np.int64)


def _kept(da, db, contract):
    """The exact sum of the kept digit products, in units of 2^(-124): by weight
    in 64 bits, then as Python integers."""
    out = 0
    for w in range(8):
        s = sum(contract(da[i], db[w - i]) for i in range(w + 1))
        out = out + s.astype(object) * (1 << (8 * (14 - w)))
    return out


def _worst(got, want):
    """max |got 2^124 - want| / |want| in units of 2^-53."""
    worst = 0.0
    for g, w in zip(got.reshape(-1), want.reshape(-1)):
        n, d = float(g).as_integer_ratio()
        worst = max(worst, abs(float((n << 124) - w * d) / d / float(w)))
    return worst / EPS


@pytest.mark.parametrize("k,n", [(64, 65), (128, 64), (129, 33), (257, 40),
                                 (1024, 64)])
def test_product_of_extreme_digits(digits, k, n):
    """Every accumulator and 64-bit sum near its largest, at depths of one to
    eight accumulation chunks: the kept sum to the result's three roundings
    (two sums joined, two scales that are powers of two, one of T2's)."""
    rng = np.random.default_rng(k)
    N = 200
    A, da = _extreme((N, k), rng, -128)
    M, dm = _extreme((k, n), rng, -126)
    Y = digits.mult(A, M)
    want = _kept(da, dm, lambda x, y: x @ y)
    assert _worst(Y, want) <= 3


@pytest.mark.parametrize("N,m", [(1024, 24), (50000, 40)])
def test_gram_of_extreme_digits(digits, N, m):
    """The same over rows: at most 152 slices, each rounded twice, added by
    eight chains of ceil(152 / 8) and eight more additions."""
    rng = np.random.default_rng(N)
    A, da = _extreme((N, m), rng, -128)
    B, db = _extreme((N, m), rng, -126)
    G = digits.gram(A, B)
    want = _kept(da, db, lambda x, y: x.T @ y)
    assert _worst(G, want) <= 2 + 19 + 8


def _localised(N, m, length):
    """Columns exp(-|i - c_j| / length) with a sign pattern: from 1 down to
    nothing over the grid, as bound states far from one another."""
    i = np.arange(N)[:, None]
    c = (np.arange(m)[None, :] + 0.5) * (N / m)
    s = np.where((i * 2654435761 >> 7) % 3 == 0, -1.0, 1.0)
    return np.asfortranarray(s * np.exp(-np.abs(i - c) / length))


@pytest.mark.parametrize("length", [20.0, 300.0])
def test_localised_columns_norm_wise(digits, length):
    """A wide range of magnitudes within a column: the Gram and the product are
    within the bound above of the exact ones, entry by entry, relative to the
    columns' largest entries. Their small entries are not good to FP64's own
    relative rounding: that is the price, and this pins what is left of it."""
    N, m, n = 20000, 16, 16
    A = _localised(N, m, length)
    B = np.roll(A, 7, axis=0)
    amax, bmax = np.abs(A).max(axis=0), np.abs(B).max(axis=0)
    G = digits.gram(A, B)
    L = np.longdouble
    exact = np.array([[np.sum(A[:, i].astype(L) * B[:, j]) for j in range(m)]
                      for i in range(m)])
    bound = (2.0 ** -58.9 * N * 4 * np.outer(amax, bmax)
             + 29 * EPS * (np.abs(A).T @ np.abs(B)))
    assert np.all(np.abs(G - exact) <= bound)
    # (the factor's columns are held against the largest of amax_k |M_kj|)
    M = ti.random_block(m, n, seed=2)
    Y = digits.mult(A, M)
    exact = A.astype(L) @ M.astype(L)
    mmax = (amax[:, None] * np.abs(M)).max(axis=0)
    bound = 2.0 ** -58.9 * m * 4 * mmax[None, :] + 3 * EPS * np.abs(exact)
    assert np.all(np.abs(Y - exact) <= bound)


def test_localised_columns_orthonormalized(digits):
    """trm_orthonormalize on the digits: orthonormal, and the oracle's block to
    rounding times the overlap's condition (about 1 here), norm-wise."""
    import paper_1108_4509_gb300 as trm
    N, m = 32768, 64
    C = _localised(N, m, 30.0)
    C /= np.linalg.norm(C, axis=0)
    t = gu.to_dev(C)
    trm.trm_orthonormalize(N, m, t.data_ptr(), gu.stream())
    got = gu.from_dev(t)
    assert np.max(np.abs(got.T @ got - np.eye(m))) < 1e-13
    assert np.max(np.abs(got - otrm.orthonormalize(C))) < 1e-13
