"""Calls at the edges of what they accept, through the C ABI: widths, padded
columns, long rows, blocks with a wide range of magnitudes."""
import ctypes as ct
import os
import subprocess
import sys

import numpy as np
import pytest

import trm_inputs as ti
from oracle import operator as op
from oracle import trm as otrm

from . import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def trm():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1108_4509_gb300 as mod
    return mod


@pytest.mark.parametrize("m", [1, 31, 32, 33, 65, 257])
def test_energy_is_the_sum_of_its_columns(trm, m):
    """E is added up by the CTA of the column sums that finishes last, from
    what the others stored: the H_D of the same call, to the rounding of m
    additions, in each of several calls with other blocks."""
    shape = (9, 8, 7)
    V = ti.gaussian_wells(shape, 4, seed=2)
    N = V.size
    opt = trm.trm_default_options(stream=gu.stream())
    h = trm.trm_create_stencil(*shape, 4, 1.0, V, m, 1e-10, opt)
    try:
        for seed in range(4):
            C = otrm.orthonormalize(ti.random_block(N, m, seed)) * (seed + 1)
            cd, g = gu.to_dev(C), gu.empty(N, m, np.float64)
            hd = gu.to_dev(np.zeros(m))
            E = trm.trm_energy_gradient(h, cd.data_ptr(), hd.data_ptr(), 0,
                                        g.data_ptr(), trm.TRM_F64, True)
            HD = gu.from_dev(hd)
            assert abs(E - HD.sum()) <= m * 2.3e-16 * np.abs(HD).sum()
    finally:
        trm.trm_destroy(h)


_FACTOR_256 = """
import numpy as np
import trm_inputs as ti
from oracle import trm as otrm
from tests import gpu_util as gu
import paper_1108_4509_gb300 as trm
N, m = 900, 256
C = ti.random_block(N, m, 7)
t = gu.to_dev(C)
trm.trm_orthonormalize(N, m, t.data_ptr(), gu.stream())
got = gu.from_dev(t)
tol = 20 * m * 2.3e-16 * np.linalg.cond(C) ** 2
assert np.max(np.abs(got.T @ got - np.eye(m))) < tol
assert np.max(np.abs(got - otrm.orthonormalize(C))) < tol
"""


def test_factor_of_256_columns_on_one_cta(trm):
    """m = 256 with the line to the blocked launches moved above it: the
    corrected factor at its largest, in a process of its own (the line is read
    once). Rounding: m eps times the overlap's condition (about 11 for this
    shape), a factor of 20 above."""
    env = dict(os.environ, TRM_CHOL_BLOCKED_FROM="300")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _FACTOR_256], cwd=root, env=env,
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("how", ["gradient", "gradient32", "iterate"])
@pytest.mark.parametrize("csr", [0, 1])
@pytest.mark.parametrize("shape,m", [((13, 11, 9), 40), ((7, 5, 3), 6),
                                     ((9, 21, 1), 20)])
def test_energy_gradient_after_an_overflow(trm, shape, m, csr, how):
    """A block that overflows leaves no trace on a handle with padded columns
    (N % 4 != 0): the next trm_energy_gradient gives E, H_D, H' and G of a
    fresh handle, byte for byte, in either type of G."""
    V = ti.gaussian_wells(shape, 4, seed=2)
    N = V.size
    assert N % 4
    opt = trm.trm_default_options(stream=gu.stream(), precond=1)

    def make():
        if csr:
            return trm.trm_create_csr(N, *ti.grid_csr(shape, 4, 1.0, V), m, 1e-10,
                                      opt)
        return trm.trm_create_stencil(*shape, 4, 1.0, V, m, 1e-10, opt)

    def energy_gradient(h, block, dt):
        g = gu.empty(N, m, [np.float32, np.float64][dt == trm.TRM_F64])
        hd, hp = gu.to_dev(np.zeros(m)), gu.empty(m, m, np.float64)
        E = trm.trm_energy_gradient(h, block.data_ptr(), hd.data_ptr(),
                                    hp.data_ptr(), g.data_ptr(), dt, True)
        return E, gu.from_dev(hd), gu.from_dev(hp), gu.from_dev(g)

    good = gu.to_dev(otrm.orthonormalize(ti.random_block(N, m, 3)))
    big = gu.to_dev(np.full((N, m), 1e200) * (1 + ti.random_block(N, m, 1)))
    types = (trm.TRM_F64, trm.TRM_F32)
    h = make()
    ref = [energy_gradient(h, good, dt) for dt in types]
    trm.trm_destroy(h)
    assert all(np.all(np.isfinite(x)) for r in ref for x in r)
    h = make()
    try:
        for k, dt in enumerate(types):
            if how == "iterate":
                trm.trm_set_block(h, big.data_ptr())
                try:
                    trm.trm_iterate(h, trm.TRM_FP64)
                except trm.TrmError:
                    pass
            else:
                energy_gradient(h, big, trm.TRM_F64 if how == "gradient"
                                else trm.TRM_F32)
            got = energy_gradient(h, good, dt)
            for a, b in zip(got, ref[k]):
                assert np.array_equal(a, b)
    finally:
        trm.trm_destroy(h)


def test_generalized_mixed_solve_on_padded_columns(trm):
    """The mixed ladder of the generalized problem on a grid with N % 4 != 0:
    the dense eigenvalues, an S-orthonormal block, and the same bytes from a
    second solve on the handle."""
    import scipy.linalg as sla
    import scipy.sparse as sp
    shape, m = (9, 11, 7), 10
    V = ti.gaussian_wells(shape, 4, seed=2)
    N = V.size
    assert N % 4
    H = op.grid_hamiltonian(shape, 4, 1.0, V)
    rp, ci, v = ti.hat_overlap_csr(shape)
    S = sp.csr_matrix((v, ci, rp), shape=(N, N))
    w = sla.eigh(H.toarray(), S.toarray(), eigvals_only=True)[:m]
    opt = trm.trm_default_options(stream=gu.stream(), precision=trm.TRM_MIXED,
                                  seed=3)
    h = trm.trm_create_stencil(*shape, 4, 1.0, V, m, 1e-10, opt)
    try:
        trm.trm_set_overlap_csr(h, rp, ci, v)
        C, D = np.zeros((N, m), order="F"), np.zeros((N, m), order="F")
        lam, _, st, status = trm.trm_solve(h, N, m, C_out=C)
        lam2, _, _, status2 = trm.trm_solve(h, N, m, C_out=D)
        assert status == 0 and status2 == 0 and st.iterations_phase[0] > 0
        assert np.array_equal(lam, lam2) and np.array_equal(C, D)
        assert np.max(np.abs(lam - w)) < 1e-9
        assert np.max(np.abs(C.T @ (S @ C) - np.eye(m))) < 1e-10
    finally:
        trm.trm_destroy(h)


@pytest.mark.parametrize("N,m", [(400, 12), (8192, 64)])
def test_block_that_cannot_be_factored_stays(trm, N, m):
    """trm_orthonormalize of a singular block returns TRM_ENOTPD and leaves the
    block as it was, the entries far below their column's largest too, on the
    FP64 products (the smaller size) and on the digits."""
    C = ti.random_block(N, m, seed=3) * 10.0 ** -np.linspace(0, 40, N)[:, None]
    C[:, m // 2] = 2.0 * C[:, 1]
    cd = gu.to_dev(C)
    with pytest.raises(trm.TrmError) as e:
        trm.trm_orthonormalize(N, m, cd.data_ptr(), gu.stream())
    assert e.value.status == -3
    assert np.array_equal(gu.from_dev(cd), C)


@pytest.mark.parametrize("csr", [0, 1])
@pytest.mark.parametrize("nx", [4, 5])
def test_most_columns_of_an_application(trm, nx, csr):
    """trm_apply_h takes 4 * 65535 columns and refuses one more, for every
    operator and type."""
    import torch
    V = np.arange(1.0, nx + 1)
    opt = trm.trm_default_options(stream=gu.stream())
    if csr:
        h = trm.trm_create_csr(nx, *ti.grid_csr((nx, 1, 1), 2, 1.0, V), 1, 1e-10,
                               opt)
    else:
        h = trm.trm_create_stencil(nx, 1, 1, 2, 1.0, V, 1, 1e-10, opt)
    H = torch.tensor(op.grid_hamiltonian((nx, 1, 1), 2, 1.0, V).toarray()).cuda()
    most = 4 * 65535
    try:
        for dt, td in ((trm.TRM_F32, torch.float32), (trm.TRM_F64, torch.float64)):
            X = torch.ones(most + 1, nx, dtype=td, device="cuda")
            Y = torch.zeros_like(X)
            trm.trm_apply_h(h, dt, X.data_ptr(), dt, Y.data_ptr(), most)
            want = (X.double() @ H)[:most]
            assert float((Y[:most].double() - want).abs().max()) < 1e-5
            with pytest.raises(trm.TrmError) as e:
                trm.trm_apply_h(h, dt, X.data_ptr(), dt, Y.data_ptr(), most + 1)
            assert e.value.status == -1
    finally:
        trm.trm_destroy(h)


def test_mp2_energy_of_a_matrix_with_long_rows(trm):
    """1500 equal entries a row: the double-float sum of a row is renormalised
    at every entry, so that its low part rounds against what one addition
    leaves and not against what all before it have. Per entry at most 2^-46.6
    of the partial sum (two low parts added, then added to the sum's), half
    the final one on average, and 2^-47 of the product: n 2^-46.6 of the sum.
    With one renormalisation at the end the errors add up in step here, and
    the energy was 7.6e-11 off."""
    n, m, v = 1500, 2, 0.7
    N = n * m
    rp = (np.arange(N + 1) * n).astype(np.int32)
    first = (np.arange(N) // n * n)[:, None]
    cols = (first + np.arange(n)[None, :]).astype(np.int32).reshape(-1)
    opt = trm.trm_default_options(stream=gu.stream())
    h = trm.trm_create_csr(N, rp, cols, np.full(N * n, v), m, 1e-10, opt)
    try:
        C = np.zeros((N, m), order="F")
        for j in range(m):
            C[j * n:(j + 1) * n, j] = 1.0 / np.sqrt(n)
        cd = gu.to_dev(C)
        trm.trm_set_block(h, cd.data_ptr())
        E, _, _ = trm.trm_iterate(h, trm.TRM_MP2)
    finally:
        trm.trm_destroy(h)
    want = m * n * n * v / n
    assert abs(E - want) <= n * 2.0 ** -46.6 * want


class _Blocks(ct.Structure):
    _fields_ = [("p", ct.c_void_p * 4), ("cols", ct.c_int), ("count", ct.c_int)]


class _GramOut(ct.Structure):
    _fields_ = [("f32", ct.c_void_p), ("split", ct.c_void_p),
                ("split_ldm", ct.c_int), ("zero_diag", ct.c_int),
                ("fine", ct.c_int)]


@pytest.mark.parametrize("N,m", [(1388, 64), (5000, 32), (36000, 64), (36000, 65),
                                 (9000, 130), (60000, 200)])
def test_fine_gram_of_positive_blocks(trm, N, m):
    """The tensor-core Gram with fine sums, all terms of one sign, where every
    truncation counts the same way: within a stage of 32 rows the sum is
    truncated by 2^-23 at a quarter, half, three quarters and the whole of its
    size (2.5 2^-23), and by the other products at 2^-10 of that. The operands'
    second terms round at 2^-22 of the value, up and down alike over the rows:
    half of that bound is more than what is left. (Chunks of eight stages are
    about 1e-6 off.)"""
    import torch
    rng = np.random.default_rng(N + m)
    A = rng.uniform(0.5, 1.0, (N, m)).astype(np.float32)
    B = rng.uniform(0.5, 1.0, (N, m)).astype(np.float32)
    a, b = gu.to_dev(A), gu.to_dev(B)
    lib = ct.CDLL(trm.LIB_PATH)
    size = lib._ZN3trm21gram_partials_doublesElii
    size.restype = ct.c_size_t
    assert lib._ZN3trm17gram_tc_fine_paysEli(ct.c_int64(N), m) & 1
    cap = size(ct.c_int64(N), m, m)
    part = torch.zeros(cap, dtype=torch.float64, device="cuda")
    out, err = gu.empty(m, m, np.float64), gu.to_dev(np.zeros(4, np.int32))
    blocks = _Blocks((ct.c_void_p * 4)(b.data_ptr(), None, None, None), m, 1)
    also = _GramOut(None, None, 0, 0, 1)
    f = lib._ZN3trm4gramIfEEbliPKT_RKNS_6BlocksIS1_EEPdS8_mP11CUstream_stPiRKNS_7GramOutE
    f(ct.c_int64(N), m, ct.c_void_p(a.data_ptr()), ct.byref(blocks),
      ct.c_void_p(out.data_ptr()), ct.c_void_p(part.data_ptr()),
      ct.c_size_t(cap), ct.c_void_p(gu.stream()), ct.c_void_p(err.data_ptr()),
      ct.byref(also))
    G = gu.from_dev(out)
    assert int(err[0]) == 0
    want = A.astype(np.float64).T @ B.astype(np.float64)
    assert np.max(np.abs(G / want - 1.0)) <= 2.5 * 2.0 ** -23 + 2.0 ** -22


@pytest.mark.parametrize("shape,m", [((13, 11, 9), 33), ((13, 11, 9), 60),
                                     ((17, 19, 21), 32), ((21, 23, 25), 40),
                                     ((31, 33, 35), 70), ((9, 21, 1), 20)])
def test_mp2_step_on_odd_grids_is_as_exact_as_multiply_adds(trm, shape, m):
    """N % 4 != 0, close to the solution: the step's own error, relative to
    the step. Grams and products of FP32 multiply-adds, or as exact: 6e-7 of
    a Gram at most (the test above) in alpha, one 6e-8 each for G, P and the
    update, a product's 2^-22: below 1e-6 in all. With the sums that other
    grids take it was 3e-6 to 8e-6."""
    order = 4
    V = ti.gaussian_wells(shape, 4, seed=6)
    N = V.size
    assert N % 4
    H = op.grid_hamiltonian(shape, order, 1.0, V)
    import scipy.sparse.linalg as spla
    w, v = (np.linalg.eigh(H.toarray()) if N < 2000 else
            spla.eigsh(H, k=m, which="SA", tol=1e-12,
                       v0=np.ones(N), ncv=4 * m))
    C = np.linalg.qr(v[:, :m] + 5e-6 * np.sqrt(3.0 / N) * 2
                     * ti.random_block(N, m, 3))[0]
    X = op.apply_h(H, C)
    HD = np.sum(C * X, axis=0)
    Xp = X - C * HD
    Hp = C.T @ Xp
    np.fill_diagonal(Hp, 0.0)
    G = -2.0 * (Xp - C @ Hp)
    B, Q, W = C.T @ G, G.T @ G, G.T @ G
    A0 = 0.5 * (Hp + Hp.T) + np.diag(HD)
    D1 = A0 @ B - B @ A0 - 0.5 * (W + W.T)
    curve = (np.sum(G * op.apply_h(H, G)) - np.sum(Q * A0)
             - np.sum((B + B.T) * D1))
    a = np.trace(W) / (2 * curve)
    Y = C + a * G
    want = np.linalg.solve(np.linalg.cholesky(Y.T @ Y), Y.T).T
    opt = trm.trm_default_options(stream=gu.stream())
    h = trm.trm_create_stencil(*shape, order, 1.0, V, m, 1e-10, opt)
    try:
        cd = gu.to_dev(C)
        trm.trm_set_block(h, cd.data_ptr())
        trm.trm_iterate(h, trm.TRM_MP2, restart=True)
        out = gu.empty(N, m, np.float64)
        trm.trm_get_block(h, out.data_ptr())
        got = gu.from_dev(out)
    finally:
        trm.trm_destroy(h)
    step = np.linalg.norm(a * G)
    assert np.linalg.norm(got - want) <= 1e-6 * step + 2.0 ** -46 * np.sqrt(m)


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("shape", [(1, 200, 1), (2, 101, 1), (3, 3, 50),
                                   (5, 5, 33), (4, 4, 40), (7, 300, 1),
                                   (9, 9, 9), (6, 11, 13), (129, 1, 1),
                                   (1, 1, 77), (1, 7, 30)])
def test_marching_stencils_of_thin_grids(trm, shape, order):
    """Planes of a few points, whose CTAs take several chunks: H C in FP32
    against the dense operator (13 terms of FP32 rounding) and the MP2 energy,
    whose H C and column dots are double-float pairs, against FP64."""
    V = ti.gaussian_wells(shape, 2, seed=2)
    N, m = V.size, 5
    H = op.grid_hamiltonian(shape, order, 1.0, V).toarray()
    C = otrm.orthonormalize(ti.random_block(N, m, seed=3))
    opt = trm.trm_default_options(stream=gu.stream())
    h = trm.trm_create_stencil(*shape, order, 1.0, V, m, 1e-10, opt)
    try:
        x32 = gu.to_dev(C, np.float32)
        y = gu.empty(N, m, np.float32)
        trm.trm_apply_h(h, trm.TRM_F32, x32.data_ptr(), trm.TRM_F32,
                        y.data_ptr(), m)
        mag = np.abs(H) @ np.abs(C)
        assert np.all(np.abs(gu.from_dev(y) - H @ C) <= 16 * 2.0 ** -24 * mag)
        cd = gu.to_dev(C)
        trm.trm_set_block(h, cd.data_ptr())
        E, _, _ = trm.trm_iterate(h, trm.TRM_MP2)
        assert abs(E - np.sum(C * (H @ C))) <= 2.0 ** -44 * np.sum(np.abs(C) * mag)
    finally:
        trm.trm_destroy(h)


@pytest.mark.parametrize("cond", [15.0, 25.0, 300.0])
@pytest.mark.parametrize("m", [33, 64, 100, 255])
def test_fp64_factor_where_the_correction_is_left_early(trm, m, cond):
    """Overlaps that the corrected FP32 factor refuses, before its products
    (a large entry of the FP32 inverse) and before it begins (two columns at a
    small angle), and one near the line: the elimination's result. Rounding: m
    eps times the condition, a factor of 20 above."""
    N = 2 * m + 100
    rng = np.random.default_rng(m)
    U = np.linalg.qr(rng.standard_normal((N, m)))[0]
    Q = np.linalg.qr(rng.standard_normal((m, m)))[0]
    C = (U * np.geomspace(1.0, cond ** 0.5, m)) @ Q
    near = C.copy()
    near[:, m - 1] = 0.9 * near[:, 3] + 0.3 * near[:, m - 1]
    for block in (C, near, C * 2.0 ** np.floor(rng.uniform(-30, 30, m))):
        ref = otrm.orthonormalize(block)
        t = gu.to_dev(block)
        trm.trm_orthonormalize(N, m, t.data_ptr(), gu.stream())
        got = gu.from_dev(t)
        unit = block / np.linalg.norm(block, axis=0)
        tol = 20 * m * 2.3e-16 * np.linalg.cond(unit) ** 2
        assert np.max(np.abs(got.T @ got - np.eye(m))) < tol
        assert np.max(np.abs(got - ref)) < tol


@pytest.mark.parametrize("gap", [1e-12, 1e-9, 1e-7, 1e-6, 1e-4])
@pytest.mark.parametrize("m", [48, 128, 200])
def test_eigenvalues_with_a_coupling_of_low_rank(trm, m, gap):
    """Diagonal blocks whose neighbours lie `gap` apart, all coupled by a matrix
    of rank one with entries just below what the FP32 sweeps rotate: its 2-norm
    is its Frobenius norm, many times what the refinement's separation takes
    for a random coupling of that size. The closing sweeps leave couplings of
    1e-13 of two diagonal entries and 1e-15 of the whole; products round at m
    eps."""
    rng = np.random.default_rng(m)
    d = np.repeat(np.linspace(1.0, 2.0, m // 8), 8)[:m]
    d = d + gap * np.arange(len(d))
    m = len(d)
    v = rng.choice([-1.0, 1.0], m)
    A = np.diag(d) + 0.9e-6 * np.linalg.norm(d) * np.outer(v, v)
    N = m + 3
    H = np.zeros((N, N))
    H[:m, :m] = A
    H[range(m, N), range(m, N)] = 9.0
    rows, cols = np.nonzero(H)
    rp = np.searchsorted(rows, np.arange(N + 1)).astype(np.int32)
    opt = trm.trm_default_options(stream=gu.stream())
    h = trm.trm_create_csr(N, rp, cols.astype(np.int32), H[rows, cols], m, 1e-10,
                           opt)
    try:
        t = gu.to_dev(np.eye(N)[:, :m])
        lam, _ = trm.trm_rayleigh_ritz(h, t.data_ptr(), m)
        C = gu.from_dev(t)
    finally:
        trm.trm_destroy(h)
    w = np.linalg.eigvalsh(A)
    scale = np.abs(w).max()
    tol = (2e-13 * np.sqrt(m) + 1e-15 * m + 20 * m * 2.3e-16) * scale
    assert np.max(np.abs(lam - w)) <= tol
    assert np.max(np.linalg.norm(H @ C - C * lam, axis=0)) <= tol
    assert np.max(np.abs(C.T @ C - np.eye(m))) <= 20 * m * 2.3e-16


@pytest.mark.parametrize("shape,m", [((13, 11, 9), 64), ((21, 23, 25), 40),
                                     ((17, 19, 21), 96), ((9, 11, 13), 260)])
def test_full_sp_rotation_on_odd_grids_does_not_shrink(trm, shape, m):
    """N % 4 != 0, tensor-core rotation, a step of some percent (so that no
    entry's change is below half a place and lost): the mean square norm of the
    columns. The entries of C before and after and the rotation's multiply-adds
    round by 2^-24 in either direction, a few 2^-24 / sqrt(N m) together; the
    overlap's small part is good to 2^-22 of its largest entry and the factor's
    diagonal is held as a pair. A truncated sum takes half a place off every
    entry, 6e-8 off the mean."""
    V = ti.gaussian_wells(shape, 4, seed=6)
    N = V.size
    assert N % 4 and N * m * m >= 5e6
    H = op.grid_hamiltonian(shape, 4, 1.0, V)
    import scipy.sparse.linalg as spla
    v = (np.linalg.eigh(H.toarray())[1] if N < 2000 else
         spla.eigsh(H, k=m, which="SA", v0=np.ones(N))[1])
    C = np.linalg.qr(v[:, :m] + 0.17 / np.sqrt(N) * ti.random_block(N, m, 3))[0]
    _, G, _, _ = otrm.energy_gradient_alg1(H, C)
    opt = trm.trm_default_options(stream=gu.stream())
    h = trm.trm_create_stencil(*shape, 4, 1.0, V, m, 1e-10, opt)
    try:
        cd = gu.to_dev(C)
        trm.trm_set_block(h, cd.data_ptr())
        _, _, a = trm.trm_iterate(h, trm.TRM_FULL_SP, restart=True)
        out = gu.empty(N, m, np.float64)
        trm.trm_get_block(h, out.data_ptr())
        got = gu.from_dev(out)
    finally:
        trm.trm_destroy(h)
    q = a * a * np.max(np.sum(G ** 2, axis=0))
    assert q > 1e-5
    bound = 16 * 2.0 ** -24 / np.sqrt(N * m) + 2.0 ** -20 * q
    assert abs(np.sum(got ** 2) / m - 1.0) <= bound


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("shape", [(9, 11, 13), (6, 5, 7), (7, 50, 1), (31, 1, 1)])
def test_fp32_stencil_of_odd_rows_operation_by_operation(trm, shape, order):
    """nx % 4 != 0: neighbours at distance one added along x, y, z, then one
    multiply-add per distance onto the rounded diagonal term. The same in numpy,
    a multiply-add through FP64 (whose second rounding differs from a true one
    in about one entry of 2^29): equal bytes."""
    V = ti.gaussian_wells(shape, 2, seed=2)
    N, m = V.size, 6
    nx, ny, nz = (tuple(shape) + (1, 1))[:3]
    f = np.float32
    C = ti.random_block(N, m, seed=3).astype(f)
    w = {2: (2.0, -1.0), 4: (2.5, -4.0 / 3.0, 1.0 / 12.0)}[order]
    ndim = sum(n > 1 for n in (nx, ny, nz))
    d = (0.5 * w[0] * ndim + V).astype(f).reshape(nz, ny, nx)
    B = C.T.reshape(m, nz, ny, nx)

    def shift(ax, k):
        pad = [(0, 0)] * 4
        pad[ax] = (abs(k), abs(k))
        take = [slice(None)] * 4
        take[ax] = slice(abs(k) + k, abs(k) + k + B.shape[ax])
        return np.pad(B, pad)[tuple(take)]

    acc = d * B
    for r in range(1, len(w)):
        s = np.zeros_like(B)
        for ax in (3, 2, 1):
            if B.shape[ax] > 1:
                s = (s + shift(ax, -r)) + shift(ax, r)
        c = np.float64(f(0.5 * w[r]))
        acc = (c * s.astype(np.float64) + acc.astype(np.float64)).astype(f)
    opt = trm.trm_default_options(stream=gu.stream())
    h = trm.trm_create_stencil(nx, ny, nz, order, 1.0, V, m - 1, 1e-10, opt)
    try:
        x = gu.to_dev(C, f)
        y = gu.empty(N, m, f)
        trm.trm_apply_h(h, trm.TRM_F32, x.data_ptr(), trm.TRM_F32, y.data_ptr(), m)
        assert np.array_equal(gu.from_dev(y), acc.reshape(m, N).T)
    finally:
        trm.trm_destroy(h)
