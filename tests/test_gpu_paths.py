"""Sequences of calls and sizes at the edges of the dispatch rules, through the
C ABI."""
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


def _near(H, m, seed):
    """An orthonormal block near the m lowest eigenvectors (its line search
    has positive curvature: the step does not depend on earlier ones)."""
    w, v = np.linalg.eigh(H.toarray())
    return np.linalg.qr(v[:, :m] + 0.01 * ti.random_block(len(w), m, seed))[0]


@pytest.mark.parametrize("mode", ["TRM_FP64", "TRM_FULL_SP", "TRM_MP2"])
@pytest.mark.parametrize("shape,m", [((13, 11, 9), 7), ((8, 8, 10), 32)])
def test_new_sequence_ignores_the_last(trm, mode, shape, m):
    """After trm_set_block or trm_rayleigh_ritz the first iteration starts a
    new CG sequence whatever G_prev and P hold: the same bytes as on a fresh
    handle, also with trm_energy_gradient in between."""
    V = ti.gaussian_wells(shape, 4, seed=2)
    N = V.size
    H = op.grid_hamiltonian(shape, 4, 1.0, V)
    cd = gu.to_dev(_near(H, m, 3))

    def first(h):
        trm.trm_set_block(h, cd.data_ptr())
        return first_iteration(h)

    def first_iteration(h):
        r = trm.trm_iterate(h, getattr(trm, mode))
        out = gu.empty(N, m, np.float64)
        trm.trm_get_block(h, out.data_ptr())
        return r, gu.from_dev(out)

    opt = trm.trm_default_options(stream=gu.stream(), precond=1)
    fresh = trm.trm_create_stencil(*shape, 4, 1.0, V, m, 1e-10, opt)
    used = trm.trm_create_stencil(*shape, 4, 1.0, V, m, 1e-10, opt)
    try:
        ref = first(fresh)
        first(used)
        trm.trm_iterate(used, getattr(trm, mode))
        again = first(used)
        assert again[0] == ref[0] and np.array_equal(again[1], ref[1])
        trm.trm_set_block(used, cd.data_ptr())
        g = gu.empty(N, m, np.float64)
        trm.trm_energy_gradient(used, cd.data_ptr(), 0, 0, g.data_ptr(),
                                trm.TRM_F64, True)
        between = first_iteration(used)
        assert between[0] == ref[0] and np.array_equal(between[1], ref[1])
        trm.trm_set_block(used, cd.data_ptr())
        other = gu.to_dev(_near(H, m, 5))
        trm.trm_rayleigh_ritz(used, other.data_ptr(), m)
        after = first_iteration(used)
        assert after[0] == ref[0] and np.array_equal(after[1], ref[1])
    finally:
        trm.trm_destroy(fresh)
        trm.trm_destroy(used)


@pytest.mark.parametrize("mode", ["TRM_FULL_SP", "TRM_MP2"])
@pytest.mark.parametrize("m", [1, 5, 31, 32, 33, 64, 65, 96, 127, 128, 129, 200,
                               255, 256, 257])
def test_step_factorisation_edges(trm, mode, m):
    """One step against (C + a G) L^{-T} element by element, at the edges of
    the 32-column panels and of the one-CTA factorisation (m = 256). The
    bound: the FP32-class gradient (dG), the FP32-class Grams of the overlap
    (dS, twice for the factor's first-order change) and the product's
    rounding, each at 2^-19 of the magnitudes multiplied, C stored in FP32 in
    full SP."""
    shape, order = (16, 12, 11), 4
    V = ti.gaussian_wells(shape, 4, seed=6)
    H = op.grid_hamiltonian(shape, order, 1.0, V)
    N = V.size
    C = otrm.orthonormalize(ti.random_block(N, m, seed=3))
    X = op.apply_h(H, C)
    Xp = X - C * np.sum(C * X, axis=0)
    Hp = C.T @ Xp
    np.fill_diagonal(Hp, 0.0)
    G = -2.0 * (Xp - C @ Hp)
    u = 2.0 ** -19
    opt = trm.trm_default_options(stream=gu.stream())
    h = trm.trm_create_stencil(*shape, order, 1.0, V, m, 1e-10, opt)
    try:
        cd = gu.to_dev(C)
        trm.trm_set_block(h, cd.data_ptr())
        _, _, a = trm.trm_iterate(h, getattr(trm, mode), restart=True)
        out = gu.empty(N, m, np.float64)
        trm.trm_get_block(h, out.data_ptr())
        C1 = gu.from_dev(out)
    finally:
        trm.trm_destroy(h)
    Y = C + a * G
    R = np.linalg.inv(np.linalg.cholesky(Y.T @ Y)).T
    f32 = 2.0 ** -24 * (np.abs(X) + np.abs(C) * np.abs(np.sum(C * X, axis=0)))
    dG = 2.0 * (f32 * (1 if mode == "TRM_FULL_SP" else 0)
                + 2.0 ** -24 * np.abs(Xp) + u * np.abs(C) @ np.abs(Hp)
                + np.abs(C) @ (u * np.abs(C).T @ np.abs(Xp)))
    cp = np.abs(C).T @ np.abs(G)
    dS = u * (a * a * np.abs(G).T @ np.abs(G) + a * (cp + cp.T))
    off = np.abs(R - np.diag(np.diag(R)))
    prod = u * np.abs(Y) @ off
    if mode == "TRM_FULL_SP":
        prod = u * np.abs(Y) @ np.abs(R)
        dS = dS + 2.0 ** -23 * np.eye(m)
    bound = (a * np.linalg.norm(dG) + 2 * np.linalg.norm(dS)
             + np.linalg.norm(prod) + 1e-12)
    assert np.linalg.norm(C1 - Y @ R) <= bound


# Grids whose size is not a multiple of four: the solver's blocks are padded.
ODD = [((13, 11, 9), 40), ((7, 5, 3), 6), ((15, 14, 13), 33), ((9, 21, 1), 20)]


@pytest.mark.parametrize("csr", [0, 1])
@pytest.mark.parametrize("shape,m", ODD)
def test_padded_columns_modes_in_turn(trm, shape, m, csr):
    """On one handle with padded columns: every mode after every other, the
    step operations in between and a start that overflows give the bytes a
    fresh handle gives."""
    V = ti.gaussian_wells(shape, 4, seed=2)
    N = V.size
    assert N % 4
    H = op.grid_hamiltonian(shape, 4, 1.0, V)
    cd = gu.to_dev(_near(H, m, 3))
    opt = trm.trm_default_options(stream=gu.stream(), precond=1)

    def make():
        if csr:
            return trm.trm_create_csr(N, *ti.grid_csr(shape, 4, 1.0, V), m, 1e-10,
                                      opt)
        nx, ny, nz = (tuple(shape) + (1, 1))[:3]
        return trm.trm_create_stencil(nx, ny, nz, 4, 1.0, V, m, 1e-10, opt)

    def two(h, mode):
        trm.trm_set_block(h, cd.data_ptr())
        r = [trm.trm_iterate(h, mode) for _ in range(2)]
        out = gu.empty(N, m, np.float64)
        trm.trm_get_block(h, out.data_ptr())
        return r, gu.from_dev(out)

    modes = [trm.TRM_FULL_SP, trm.TRM_FP64, trm.TRM_MP2]
    ref = {}
    for md in modes:
        h = make()
        ref[md] = two(h, md)
        trm.trm_destroy(h)
    h = make()
    try:
        g = gu.empty(N, m, np.float64)
        big = gu.to_dev(np.full((N, m), 1e200) * (1 + ti.random_block(N, m, 1)))
        for k, md in enumerate(modes + modes[::-1] + [trm.TRM_FP64]):
            r, C = two(h, md)
            assert r == ref[md][0] and np.array_equal(C, ref[md][1]), (k, md)
            if k % 3 == 0:
                trm.trm_energy_gradient(h, cd.data_ptr(), 0, 0, g.data_ptr(),
                                        trm.TRM_F64, True)
            elif k % 3 == 1:
                other = gu.to_dev(_near(H, m, 5))
                trm.trm_rayleigh_ritz(h, other.data_ptr(), m)
            else:
                trm.trm_set_block(h, big.data_ptr())
                try:
                    trm.trm_iterate(h, md)
                except trm.TrmError:
                    pass
    finally:
        trm.trm_destroy(h)


@pytest.mark.parametrize("shape,m", ODD)
def test_padded_columns_solve(trm, shape, m):
    """A mixed solve on padded columns from a host block, the block returned to
    the host and to the device: the oracle's eigenvalues, the same bytes."""
    V = ti.gaussian_wells(shape, 4, seed=2)
    N = V.size
    H = op.grid_hamiltonian(shape, 4, 1.0, V)
    w = np.linalg.eigvalsh(H.toarray())[:m]
    C0 = np.asfortranarray(_near(H, m, 3))
    nx, ny, nz = (tuple(shape) + (1, 1))[:3]
    opt = trm.trm_default_options(stream=gu.stream())
    h = trm.trm_create_stencil(nx, ny, nz, 4, 1.0, V, m, 1e-10, opt)
    try:
        Ch = np.zeros((N, m), order="F")
        lam, eg, _, status = trm.trm_solve(h, N, m, C_out=Ch, C0=C0)
        assert status == 0
        cd = gu.empty(N, m, np.float64)
        lam2, _, _, status2 = trm.trm_solve(h, N, m, C_out=cd.data_ptr(),
                                            C_on_device=True, C0=C0)
        assert status2 == 0 and np.array_equal(lam, lam2)
        assert np.array_equal(gu.from_dev(cd), Ch)
        assert np.max(np.abs(lam - w)) < 1e-9
        assert np.max(np.abs(Ch.T @ Ch - np.eye(m))) < 1e-12
        assert np.max(np.abs(op.apply_h(H, Ch) - Ch * lam)) < 1e-8
    finally:
        trm.trm_destroy(h)


@pytest.mark.parametrize("N,m", [(500009, 8), (20001, 63), (20002, 64),
                                 (20003, 65), (6000, 127), (6000, 128),
                                 (6001, 129), (3000, 200), (1031, 256),
                                 (1024, 300)])
def test_digit_products_orthonormalize(trm, N, m):
    """Fig. ONFIG through the digit Gram and product at the edges of their
    128 x 64 tiles and 32-row stages. Columns of very different size are
    scaled one by one, so they cost no accuracy: the result is that of the
    unscaled columns to rounding times the condition of the overlap (at most
    a few for random columns of these shapes; 40 with m = N / 4)."""
    C = ti.random_block(N, m, seed=4)
    scale = 10.0 ** np.linspace(-15, 15, m)
    ref = otrm.orthonormalize(C)
    for block in (C, C * scale):
        cd = gu.to_dev(block)
        trm.trm_orthonormalize(N, m, cd.data_ptr(), gu.stream())
        got = gu.from_dev(cd)
        assert np.max(np.abs(got.T @ got - np.eye(m))) < 1e-13
        assert np.max(np.abs(got - ref)) < 1e-13


def test_digit_products_constant_and_non_finite(trm):
    """The integer sums at their largest (equal entries, all digits at an
    extreme), a zero column, and an infinity or NaN, which must not vanish."""
    N, m = 8192, 64
    x = np.nextafter(1.0, 0.0)
    C = np.zeros((N, m), order="F")
    step = N // m
    for j in range(m):  # orthogonal: one constant stretch per column
        C[j * step:(j + 1) * step, j] = x * 2.0 ** (j - 30)
    cd = gu.to_dev(C)
    trm.trm_orthonormalize(N, m, cd.data_ptr(), gu.stream())
    got = gu.from_dev(cd)
    ref = (C != 0) / np.sqrt(step)
    assert np.max(np.abs(got - ref)) < 1e-15
    one = np.full((N, 8), x)
    one[:, 1:] *= (np.arange(N)[:, None] % np.arange(2, 9) == 0)
    wide = np.concatenate([one] + [ti.random_block(N, 56, seed=2)], axis=1)
    cd = gu.to_dev(wide)
    trm.trm_orthonormalize(N, m, cd.data_ptr(), gu.stream())
    assert np.max(np.abs(gu.from_dev(cd) - otrm.orthonormalize(wide))) < 1e-12
    for bad in (np.inf, np.nan, 0.0):
        D = np.array(wide, order="F")
        if bad == 0.0:
            D[:, 5] = 0.0
        else:
            D[77, 5] = bad
        cd = gu.to_dev(D)
        with pytest.raises(trm.TrmError) as e:
            trm.trm_orthonormalize(N, m, cd.data_ptr(), gu.stream())
        assert e.value.status == -3


@pytest.mark.parametrize("shape,m", [((15, 14, 13), 200), ((16, 16, 12), 130),
                                     ((31, 33, 35), 33)])
def test_digit_products_fp64_step(trm, shape, m):
    """One FP64 iteration whose contractions run on digits, against the same
    step formed in FP64 on the host: rounding times the magnitudes involved."""
    V = ti.gaussian_wells(shape, 4, seed=6)
    H = op.grid_hamiltonian(shape, 4, 1.0, V)
    N = V.size
    C = otrm.orthonormalize(ti.random_block(N, m, seed=3))
    E0, G0, _, _ = otrm.energy_gradient_alg1(H, C)
    opt = trm.trm_default_options(stream=gu.stream(), precision=trm.TRM_FP64)
    h = trm.trm_create_stencil(*shape, 4, 1.0, V, m, 1e-10, opt)
    try:
        cd = gu.to_dev(C)
        trm.trm_set_block(h, cd.data_ptr())
        E, r, a = trm.trm_iterate(h, trm.TRM_FP64)
        out = gu.empty(N, m, np.float64)
        trm.trm_get_block(h, out.data_ptr())
        C1 = gu.from_dev(out)
    finally:
        trm.trm_destroy(h)
    assert E == pytest.approx(E0, rel=1e-13)
    assert r == pytest.approx(otrm.rms_residual(G0), rel=1e-12)
    Y = C + a * G0
    L = np.linalg.cholesky(Y.T @ Y)
    assert np.max(np.abs(C1 - np.linalg.solve(L, Y.T).T)) < 1e-12


@pytest.mark.parametrize("side", [-1, 1])
@pytest.mark.parametrize("m", [1, 7, 8, 9, 160, 161])
def test_polar_factor_on_both_sides_of_its_rule(trm, m, side):
    """||M^T M - I||_F a little below 1/2 takes Newton-Schulz steps, above it
    the eigensolver: both give the oracle's extrapolation. The sizes lie at the
    edges of the products' tiles. Rounding: m eps in each of some ten products
    of matrices of norm up to 2."""
    N = 2 * m + 50
    rng = np.random.default_rng(m)
    full = np.linalg.qr(rng.standard_normal((N, 2 * m)))[0]
    q1 = np.linalg.qr(rng.standard_normal((m, m)))[0]
    q2 = np.linalg.qr(rng.standard_normal((m, m)))[0]
    d = rng.uniform(0.2, 1.0, m)  # 1 - cos^2 of the principal angles
    d *= (0.5 + side * 1e-3) / np.linalg.norm(d)
    C0 = full[:, :m]
    C1 = (C0 @ q1 * np.sqrt(1 - d) + full[:, m:] * np.sqrt(d)) @ q2
    want = otrm.extrapolate(C0, C1, 1.0)
    d0, d1 = gu.to_dev(C0), gu.to_dev(C1)
    dn = gu.empty(N, m, np.float64)
    trm.trm_extrapolate(N, m, d0.data_ptr(), d1.data_ptr(), 1.0, dn.data_ptr(),
                        gu.stream())
    assert np.max(np.abs(gu.from_dev(dn) - want)) < 20 * m * 2.3e-16 + 1e-14


@pytest.mark.parametrize("cond", [4.0, 1e4])
@pytest.mark.parametrize("m", [32, 33, 64, 129, 255, 256])
def test_fp64_factor_corrected_and_eliminated(trm, m, cond):
    """C^T C of condition 4 takes the corrected FP32 factor (33 <= m < 256), of
    condition 1e4 the FP64 elimination behind it; the columns' scales span
    2^+-40, which the factor's scaling takes out. Rounding of the Gram matrix
    and the factor: m eps times the condition, a factor of 20 above."""
    N = 2 * m + 100
    rng = np.random.default_rng(m)
    U = np.linalg.qr(rng.standard_normal((N, m)))[0]
    V = np.linalg.qr(rng.standard_normal((m, m)))[0]
    s = np.geomspace(1.0, cond ** 0.5, m)
    C = (U * s) @ V * 2.0 ** np.floor(rng.uniform(-40, 40, m))
    ref = otrm.orthonormalize(C)
    t = gu.to_dev(C)
    trm.trm_orthonormalize(N, m, t.data_ptr(), gu.stream())
    got = gu.from_dev(t)
    tol = 20 * m * 2.3e-16 * cond
    assert np.max(np.abs(got.T @ got - np.eye(m))) < tol
    assert np.max(np.abs(got - ref)) < tol
