"""The calls whose speed is measured, through the library's public entry points.

A case is a dict of plain values; its "do" names the call:

  iterate      trm_set_block, `steps` times trm_iterate, trm_get_block: the
               block iteration itself in one precision mode
  solve        trm_solve of one problem from a random block
  serve        a batch of requests through the request server
  extrapolate  trm_extrapolate: the next block of a chain of problems
  ritz         trm_rayleigh_ritz on a block close to the solution

Potentials are separable, V = vx(x) + vy(y) + vz(z) with each profile a sum of
Gaussian wells, so that H's eigenpairs are sums and products of 1-D ones: blocks
at any distance from the solution are made in milliseconds, and the exact
eigenvalues of every solve are known. The kernels take the same path for them as
for any other potential.
"""
import math
import random

import numpy as np
import torch

import paper_1108_4509_gb300 as trm
import trm_inputs

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # A small problem start to finish (16^3 grid, m = 16): launches and
        # latency, not bandwidth, make its time.
        dict(name="solve_grid16_m16", do="solve", nx=16, ny=16, nz=16, order=2,
             wells=3, m=16, precond=0, tol=1e-10, iters=210),
        # The benchmark's problem size (48^3, 13-point, m = 128, diagonal M).
        dict(name="solve_grid48_m128", do="solve", nx=48, ny=48, nz=48, order=4,
             wells=8, m=128, precond=1, tol=1e-10, iters=1100),
        # Independent requests of the serving mix (12^3..40^3, m = 8..96).
        dict(name="serve_16_requests", do="serve", requests=16, mix=1, n_lo=12,
             n_hi=40, m_lo=8, m_hi=96, tol=1e-8, iters=390),
        # The bulk of a mixed solve: full single precision, then MP2.
        dict(name="sp_grid48_m128", do="iterate", mode="sp", nx=48, ny=48, nz=48,
             order=4, wells=8, m=128, precond=1, csr=0, steps=2),
        dict(name="mp2_grid48_m128", do="iterate", mode="mp2", nx=48, ny=48,
             nz=48, order=4, wells=8, m=128, precond=1, csr=0, steps=2),
        # The large problem (96^3, m = 512): dense contractions dominate.
        dict(name="mp2_grid96_m512", do="iterate", mode="mp2", nx=96, ny=96,
             nz=96, order=4, wells=16, m=512, precond=1, csr=0, steps=2),
        # An odd grid and block width, as half of the serving mix has them.
        dict(name="sp_grid39x41x37_m90", do="iterate", mode="sp", nx=39, ny=41,
             nz=37, order=4, wells=7, m=90, precond=0, csr=0, steps=2),
        # The paper's own operator: the 2-D Dirichlet Laplacian, 192^2, m = 220.
        dict(name="mp2_laplace192_m220", do="iterate", mode="mp2", nx=192,
             ny=192, nz=1, order=2, wells=0, m=220, precond=0, csr=0, steps=2),
        # The operator handed over as an explicit sparse matrix.
        dict(name="mp2_csr48_m128", do="iterate", mode="mp2", nx=48, ny=48,
             nz=48, order=4, wells=8, m=128, precond=0, csr=1, steps=2),
        # The all-FP64 mode.
        dict(name="fp64_grid48_m128", do="iterate", mode="fp64", nx=48, ny=48,
             nz=48, order=4, wells=8, m=128, precond=1, csr=0, steps=2),
        # Chains of related problems: the next starting block.
        dict(name="extrapolate_grid32_m48", do="extrapolate", nx=32, ny=32,
             nz=32, order=4, wells=6, m=48),
        # The closing diagonalisation.
        dict(name="ritz_grid32_m64", do="ritz", nx=32, ny=32, nz=32, order=4,
             wells=6, m=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: grid edges 8..96 (2-D: 24..256), m 4..512,
    both stencil orders, stencil and CSR, every mode."""
    do = rng.choice(["iterate"] * 6 + ["solve", "serve", "extrapolate", "ritz"])
    order = rng.choice([2, 4])
    if do == "serve":
        lo = rng.randint(10, 16)
        return dict(do="serve", requests=rng.randint(6, 14),
                    mix=rng.randint(2, 1 << 20), n_lo=lo,
                    n_hi=rng.randint(lo + 8, 36), m_lo=rng.randint(4, 12),
                    m_hi=rng.randint(24, 80), tol=1e-8, iters=390)
    # the most m^2 N a call may take: the largest listed iterations; the
    # FP64 calls and the whole solves stay below their listed ones
    limit = 96 ** 3 * 512 ** 2
    mode = rng.choice(["sp", "sp", "mp2", "mp2", "fp64"])
    if do == "iterate" and mode == "fp64" or do in ("extrapolate", "ritz"):
        limit = 48 ** 3 * 128 ** 2
    elif do == "solve":
        limit = 32 ** 3 * 64 ** 2
    two_d = do == "iterate" and rng.random() < 0.2
    edges = (24, 256, 2) if two_d else (8, 96, 3)
    while True:
        n = [_log_int(rng, edges[0], edges[1]) for _ in range(edges[2])]
        N = math.prod(n)
        m = _log_int(rng, 4, 512)
        if m * 8 <= N and N * m * m <= limit and N * m <= 96 ** 3 * 512:
            break
    nx, ny, nz = (n + [1])[:3]
    c = dict(do=do, nx=nx, ny=ny, nz=nz, order=order,
             wells=max(2, min(n) // 6), m=m)
    if do == "solve":
        c.update(precond=rng.choice([0, 1]), tol=1e-10, iters=400)
    if do == "iterate":
        csr = int(rng.random() < 0.2 and N <= 48 ** 3)
        c.update(mode=mode, precond=rng.choice([0, 1]), csr=csr, steps=2)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_AXIS = {2: (2.0, -1.0), 4: (2.5, -4.0 / 3.0, 1.0 / 12.0)}


class _Problem:
    """A separable H on a Dirichlet grid with h = 1, and its 1-D eigenpairs."""

    def __init__(self, shape, order, wells, rng):
        self.shape, self.order = shape, order
        self.N = math.prod(shape)
        axes = [n for n in shape if n > 1]
        self.v = []
        for n in shape:
            x = np.arange(n)
            v = np.zeros(n)
            if n > 1:
                for _ in range(wells):
                    d = rng.uniform(-2.0, -0.5) / len(axes)
                    v += d * np.exp(-((x - rng.uniform(0, n - 1)) ** 2) / 4.5)
            self.v.append(v)
        vx, vy, vz = self.v
        self.V = (vz[:, None, None] + vy[None, :, None] + vx).reshape(-1)
        self.vals, self.vecs = [], []
        for n, v in zip(shape, self.v):
            a = np.diag(v.copy())
            if n > 1:
                for k, w in enumerate(_AXIS[order]):
                    e = np.full(n - k, 0.5 * w)
                    a += np.diag(e) if k == 0 else np.diag(e, k) + np.diag(e, -k)
            w, u = np.linalg.eigh(a)
            self.vals.append(w)
            self.vecs.append(u)
        sums = (self.vals[2][:, None, None] + self.vals[1][None, :, None]
                + self.vals[0]).reshape(-1)
        self.rank = np.argsort(sums, kind="stable")
        self.sums = sums[self.rank]

    def vectors(self, ranks):
        """Eigenvectors of the given ranks as a (len, N) FP64 device tensor."""
        nx, ny, _ = self.shape
        g = self.rank[np.asarray(ranks)]
        i = (g % nx, (g // nx) % ny, g // (nx * ny))
        x, y, z = (torch.as_tensor(np.ascontiguousarray(u[:, k].T), device=DEV)
                   for u, k in zip(self.vecs, i))
        return (z[:, :, None, None] * y[:, None, :, None]
                * x[:, None, None, :]).reshape(len(g), self.N)

    def near(self, m, far, seed):
        """An orthonormal block (m, N): the m lowest eigenvectors, each turned
        by an angle of about `far` towards a higher one, and mixed."""
        rng = np.random.RandomState(seed & 0x7FFFFFFF)
        top = min(self.N, 6 * m)
        other = m + rng.permutation(top - m)[:m]
        th = torch.as_tensor(far * rng.uniform(0.3, 1.0, m), device=DEV)
        C = self.vectors(np.arange(m)).mul_(torch.cos(th)[:, None])
        C += self.vectors(other).mul_(torch.sin(th)[:, None])
        q = np.eye(m) + far * rng.standard_normal((m, m)) / math.sqrt(m)
        q = torch.as_tensor(np.linalg.qr(q)[0], device=DEV)
        return q @ C


def _shape(case):
    return case["nx"], case["ny"], case["nz"]


def _problem(case, seed):
    return _Problem(_shape(case), case["order"], case["wells"],
                    random.Random(seed))


def _solvable(shape, order, wells, m, gap, rng):
    """A problem whose wanted eigenvalues are separated, so that it converges
    in a usual number of iterations and its vectors are defined."""
    while True:
        p = _Problem(shape, order, wells, rng)
        d = np.diff(p.sums[:m + 1])
        if d[-1] >= gap and d.min() >= gap / 200:
            return p
        gap *= 0.97


_MODE = {"sp": trm.TRM_FULL_SP, "mp2": trm.TRM_MP2, "fp64": trm.TRM_FP64}
# distance from the solution: full SP does the bulk, MP2 the last digits
_FAR = {"sp": 0.05, "mp2": 5e-6, "fp64": 1e-3}


def _requests(case, seed):
    mix = random.Random(case["mix"])
    rng = random.Random(seed)
    got = []
    for _ in range(case["requests"]):
        n = mix.randint(case["n_lo"], case["n_hi"])
        order = mix.choice([2, 4])
        m = mix.randint(case["m_lo"], case["m_hi"])
        got.append((_solvable((n, n, n), order, max(2, n // 6), m, 5e-3, rng),
                    m, rng.randrange(1 << 30)))
    return got


class _Server:
    def __init__(self):
        self.handle = trm.trm_server_create(64 << 30, 16)

    def __del__(self):
        trm.trm_server_destroy(self.handle)


def _solver(p, m, tol, stream, csr=0, **opts):
    if csr:
        rowptr, cols, vals = trm_inputs.grid_csr(p.shape, p.order, 1.0, p.V)
        return trm.Solver.csr(p.N, rowptr, cols, vals, m, tol, stream=stream,
                              **opts)
    return trm.Solver.stencil(p.shape, p.order, 1.0, p.V, m, tol, stream=stream,
                              **opts)


def prepare(case, seed):
    do = case["do"]
    if do == "serve":
        return dict(do=do, server=_Server(), tol=case["tol"],
                    requests=_requests(case, seed))
    stream = torch.cuda.Stream()
    s = dict(do=do, stream=stream, m=case["m"])
    m, raw = case["m"], stream.cuda_stream
    if do == "solve":
        p = _solvable(_shape(case), case["order"], case["wells"], m, 2e-3,
                      random.Random(seed))
        s["solver"] = _solver(p, m, case["tol"], raw, precond=case["precond"],
                              seed=seed)
        s["C"] = torch.empty(m, p.N, dtype=F64, device=DEV)
    else:
        p = _problem(case, seed)
        if do == "iterate":
            s["mode"], s["steps"] = case["mode"], case["steps"]
            s["C0"] = p.near(m, _FAR[case["mode"]], seed)
            s["solver"] = _solver(p, m, 1e-10, raw, csr=case["csr"],
                                  precision=_MODE[case["mode"]],
                                  precond=case["precond"])
        elif do == "extrapolate":
            s["prev"], s["cur"] = p.near(m, 0.02, seed), p.near(m, 0.01, seed + 1)
        elif do == "ritz":
            s["C0"] = p.near(m, 1e-3, seed)
            s["solver"] = _solver(p, m, 1e-10, raw, precision=trm.TRM_FP64)
    s["N"] = p.N
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
def run(s):
    if s["do"] == "serve":
        srv = s["server"].handle
        tickets = [trm.trm_server_submit(srv, p.shape, p.order, 1.0, p.V, m,
                                         s["tol"],
                                         trm.trm_default_options(seed=seed))
                   for p, m, seed in s["requests"]]
        out = []
        for t, (_, m, _) in zip(tickets, s["requests"]):
            lam, eg, _, status, _ = trm.trm_server_wait(srv, t, m)
            if status != 0:
                raise RuntimeError("a request ended with status %d" % status)
            out.append({"lam": lam, "E_G": eg})
        return out
    with torch.cuda.stream(s["stream"]):
        return _run_on(s)


def _run_on(s):
    N, m = s["N"], s["m"]
    if s["do"] == "extrapolate":
        out = torch.empty(m, N, dtype=F64, device=DEV)
        trm.trm_extrapolate(N, m, s["prev"].data_ptr(), s["cur"].data_ptr(), 1.0,
                            out.data_ptr(), s["stream"].cuda_stream)
        return out
    h = s["solver"].handle
    if s["do"] == "solve":
        lam, eg, _, status = trm.trm_solve(h, N, m, C_out=s["C"].data_ptr(),
                                           C_on_device=True)
        if status != 0:
            raise RuntimeError("the solve ended with status %d" % status)
        # the vectors of a solve stopped at a residual of 1e-10 are defined to
        # about 1e-10 / gap: they are handed on in single precision
        return {"lam": lam, "E_G": eg, "C": s["C"].float()}
    if s["do"] == "ritz":
        C = s["C0"].clone()
        lam, res = trm.trm_rayleigh_ritz(h, C.data_ptr(), m)
        return {"lam": lam, "res": res, "C": C}
    mode = _MODE[s["mode"]]
    C = torch.empty(m, N, dtype=F64, device=DEV)
    trm.trm_set_block(h, s["C0"].data_ptr())
    # (the residual norm and the step length, which the call also returns,
    # steer the iteration; the energies and the block are its results)
    E = [trm.trm_iterate(h, mode)[0] for _ in range(s["steps"])]
    trm.trm_get_block(h, C.data_ptr())
    # full single precision holds C in FP32: so does the program after it
    return {"C": C.float() if s["mode"] == "sp" else C, "E": E}


def work(case):
    """Bytes and flops a pass cannot do without. Per iteration: C, G and P read
    and written once, the potential once, and the dense products at 10 m^2 N
    (H' 2, the three line-search products 5, gradient 2, triangular rotation 1).
    A solve is taken at its usual number of iterations."""
    if case["do"] == "serve":
        mix, b, f = random.Random(case["mix"]), 0.0, 0.0
        for _ in range(case["requests"]):
            N = float(mix.randint(case["n_lo"], case["n_hi"])) ** 3
            mix.choice([2, 4])
            m = mix.randint(case["m_lo"], case["m_hi"])
            b += case["iters"] * (24.0 * N * m + 8 * N)
            f += case["iters"] * 10.0 * m * m * N
        return {"bytes": b, "flops": f}
    N = float(case["nx"] * case["ny"] * case["nz"])
    m = case["m"]
    if case["do"] == "extrapolate":
        return {"bytes": 24.0 * N * m, "flops": 7.0 * m * m * N}
    if case["do"] == "ritz":
        return {"bytes": 16.0 * N * m + 8 * N, "flops": 8.0 * m * m * N}
    steps = case.get("steps", case.get("iters"))
    size = {"sp": 24.0, "mp2": 32.0, "fp64": 48.0}[case.get("mode", "sp")]
    by = steps * (size * N * m + 8 * N)
    if case.get("csr"):
        by += steps * 13 * 12.0 * N
    return {"bytes": by, "flops": steps * 10.0 * m * m * N}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _apply(p, C):
    """H C for C of shape (m, N)."""
    nx, ny, nz = p.shape
    B = C.reshape(-1, nz, ny, nx)
    w = _AXIS[p.order]
    dims = [d for d, n in ((3, nx), (2, ny), (1, nz)) if n > 1]
    diag = torch.as_tensor(p.V.reshape(nz, ny, nx) + 0.5 * w[0] * len(dims),
                           device=DEV)
    X = B * diag
    for d in dims:
        n = B.shape[d]
        for k in range(1, len(w)):
            X.narrow(d, 0, n - k).add_(B.narrow(d, k, n - k), alpha=0.5 * w[k])
            X.narrow(d, k, n - k).add_(B.narrow(d, 0, n - k), alpha=0.5 * w[k])
    return X.reshape(C.shape), diag.reshape(-1)


def _ortho(C):
    """Rows made orthonormal by the Cholesky factor of their Gram matrix."""
    L = torch.linalg.cholesky(C @ C.T)
    return torch.linalg.solve_triangular(L, C, upper=False)


def _iterate64(p, C, steps, precond):
    """`steps` conjugate-gradient steps of trace minimization in FP64: the
    energy and gradient, the Polak-Ribiere direction, the minimiser of the
    energy's second-order expansion along it, and orthonormalization."""
    m = C.shape[0]
    P = Gp = a_prev = None
    energies = []
    for _ in range(steps):
        X, diag = _apply(p, C)
        HD = (C * X).sum(1)
        X -= HD[:, None] * C
        Hp = C @ X.T
        Hp.fill_diagonal_(0.0)
        G = (X - Hp.T @ C).mul_(-2.0)
        del X
        MG = G / (diag - diag.min() + 1.0) if precond else G
        gmg = (G * MG).sum()
        gamma = 0.0
        if P is not None:
            gamma = float((gmg - (Gp * MG).sum()) / a_prev)
            if not float(gmg) + gamma * float((G * P).sum()) > 0.0:
                gamma = 0.0
        P = MG + gamma * P if gamma else MG.clone()
        a_prev, Gp = gmg, G
        B, Q, W = C @ P.T, P @ P.T, P @ G.T
        php = (P * _apply(p, P)[0]).sum()
        A0 = 0.5 * (Hp + Hp.T) + torch.diag(HD)
        D1 = A0 @ B - B @ A0 - 0.5 * (W + W.T)
        slope = -float(W.trace())
        curve = float(php - (Q * A0).sum() - ((B + B.T) * D1).sum())
        alpha = min(-slope / (2 * curve), math.sqrt(m / float(Q.trace())))
        energies.append(float(HD.sum()))
        C = _ortho(C + alpha * P)
    return {"C": C, "E": energies}


def _sign(C):
    """Each row's entry of largest magnitude made positive."""
    top = C.gather(1, C.abs().argmax(1, keepdim=True))
    return C * torch.sign(top)


def exact(case, seed):
    do = case["do"]
    if do == "serve":
        return [{"lam": p.sums[:m], "E_G": float(p.sums[:m].sum())}
                for p, m, _ in _requests(case, seed)]
    m = case["m"]
    if do == "solve":
        p = _solvable(_shape(case), case["order"], case["wells"], m, 2e-3,
                      random.Random(seed))
        return {"lam": p.sums[:m], "E_G": float(p.sums[:m].sum()),
                "C": _sign(p.vectors(np.arange(m)))}
    p = _problem(case, seed)
    if do == "extrapolate":
        prev, cur = p.near(m, 0.02, seed), p.near(m, 0.01, seed + 1)
        u, _, vt = torch.linalg.svd(prev @ cur.T)
        return _ortho(2.0 * cur - (u @ vt).T @ prev)
    if do == "ritz":
        C = p.near(m, 1e-3, seed)
        A = C @ _apply(p, C)[0].T
        lam, z = torch.linalg.eigh(0.5 * (A + A.T))
        C = _sign(z.T @ C)
        res = (_apply(p, C)[0] - lam[:, None] * C).norm(dim=1)
        return {"lam": lam, "res": res, "C": C}
    return _iterate64(p, p.near(m, _FAR[case["mode"]], seed), case["steps"],
                      case["precond"])
