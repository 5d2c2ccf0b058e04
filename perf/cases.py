"""The work a user of this library has it do, as cases that can be timed and
compared: the vector calls, the sparse product, the three Krylov methods, the
mixed-precision solve, the batched frequency sweep and one step of a
sound-speed inversion, from a 20x20x20 box to a 200x100x80 cavity.

Matrices are Q1 (trilinear hexahedral) Helmholtz matrices on a box of cubic
elements, A = K - w^2 M_c + i w B_c, with a sound speed drawn per element,
u = 0 on the bottom face and an impedance condition on the top one, built here
with torch on the GPU; one case has ragged random rows instead.

Solves run to convergence, to a tolerance at which the solution is settled
whatever the rounding on the way (the iterates are not: BiCGStab magnifies a
last-bit difference to the size of x within some ten iterations).  On the
large meshes the frequency is low enough (points per wavelength, `ppw`) for a
solve to take about a second; an iteration costs the same at any frequency.
"""
import itertools
import math

import numpy as np
import torch

import paper_2112_11880_gb300 as helm
from paper_2112_11880_gb300 import autograd as hgrad

DEV = "cuda"
C0 = 340.0  # m/s


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the vector calls of a Krylov iteration written by hand on the unit
        # box (9,261 unknowns): launches and latency
        {"name": "blas1_box20", "kind": "blas1", "n": 9261, "dtype": "c128"},
        # the same calls at a length of the paper's tables
        {"name": "blas1_9m", "kind": "blas1", "n": 9_000_000, "dtype": "c128"},
        # a general CSR matrix: complex entries, rows of 0 to 60 entries in
        # random columns, no structure to use
        {"name": "spmv_ragged", "kind": "spmv_ragged", "n": 20011, "max_row": 60, "dtype": "c128"},
        # the product on the car-cavity mesh (376,431 unknowns)
        {"name": "spmv_cavity120", "kind": "spmv", "nx": 120, "ny": 60, "nz": 50, "ppw": 10.0, "dtype": "c128"},
        # the complex64 product on the mesh of the mixed-precision runs
        # (1.64 M unknowns)
        {"name": "spmv64_cavity200", "kind": "spmv", "nx": 200, "ny": 100, "nz": 80, "ppw": 10.0, "dtype": "c64"},
        # BiCGStab on the unit box at 1500 Hz: small, thousands of
        # iterations, each a handful of tiny kernels
        {"name": "solve_box20", "kind": "solve", "method": "bicgstab", "nx": 20, "ny": 20, "nz": 20, "ppw": 4.533,
         "tol": 1e-12},
        # the benchmark's method and mesh, at 340 Hz (h = 0.025)
        {"name": "bicgstab_cavity120", "kind": "solve", "method": "bicgstab", "nx": 120, "ny": 60, "nz": 50,
         "ppw": 40.0, "tol": 1e-11},
        # the fastest of the paper's methods there, BiCGStab(4)
        {"name": "bicgstab4_cavity120", "kind": "solve", "method": "bicgstabl", "nx": 120, "ny": 60, "nz": 50,
         "ppw": 30.0, "tol": 1e-11},
        # TFQMR on the mesh of the gradient runs (109,593 unknowns)
        {"name": "tfqmr_80", "kind": "solve", "method": "tfqmr", "nx": 80, "ny": 40, "nz": 32, "ppw": 15.0,
         "tol": 1e-11},
        # complex64 inner solves under FP64 refinement, to convergence
        {"name": "mixed_60", "kind": "mixed", "nx": 60, "ny": 30, "nz": 25, "ppw": 10.0, "tol": 1e-11},
        # the frequency response of a cavity: 64 frequencies on one mesh
        {"name": "sweep60", "kind": "sweep", "nx": 60, "ny": 30, "nz": 25, "freqs": 64, "fmin": 50.0, "fmax": 300.0,
         "tol": 1e-10},
        # one step of a sound-speed inversion: assembly, forward solve, loss at
        # receivers, adjoint solve, gradient per element
        {"name": "inversion_30", "kind": "inversion", "nx": 30, "ny": 15, "nz": 12, "ppw": 10.0, "tol": 1e-12},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi):
    """A box of about lo..hi nodes: the longest side first, any remainders."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ry, rz = rng.uniform(0.4, 1.0), rng.uniform(0.35, 1.0)
    nx = (n / (ry * rz)) ** (1 / 3)
    return {"nx": max(3, int(nx)), "ny": max(3, int(nx * ry)), "nz": max(3, int(nx * rz))}


def draw(rng):
    kind = rng.choice(["blas1", "spmv", "spmv", "spmv_ragged", "solve", "solve", "solve", "mixed", "sweep",
                       "inversion"])
    ppw = round(rng.uniform(10.0, 15.0), 3)
    if kind == "blas1":
        return {"kind": kind, "n": _log(rng, 2000, 9_000_000), "dtype": rng.choice(["c128", "c128", "c64"])}
    if kind == "spmv_ragged":
        return {"kind": kind, "n": _log(rng, 3000, 200_000), "max_row": rng.randint(8, 60),
                "dtype": rng.choice(["c128", "c64"])}
    if kind == "spmv":
        return {"kind": kind, **_box(rng, 4000, 390_000), "ppw": ppw, "dtype": rng.choice(["c128", "c64"])}
    if kind == "solve":
        box = _box(rng, 2000, 370_000)
        if box["nx"] > 55:
            ppw = round(3.3 * ppw, 3)  # low frequencies on the large meshes
        return {"kind": kind, "method": rng.choice(sorted(_METHODS)), **box, "ppw": ppw, "tol": 1e-11}
    if kind == "mixed":
        return {"kind": kind, **_box(rng, 6000, 40_000), "ppw": ppw, "tol": 1e-11}
    if kind == "sweep":
        return {"kind": kind, **_box(rng, 4000, 40_000), "freqs": rng.randint(5, 64), "fmin": 50.0, "fmax": 300.0,
                "tol": 1e-10}
    return {"kind": kind, **_box(rng, 2000, 6500), "ppw": ppw, "tol": 1e-12}


# ---------------------------------------------------------------- problems

def _elements(h):
    """Element stiffness, mass and top-face mass, local node ax + 2 ay + 4 az."""
    k1 = np.array([[1.0, -1.0], [-1.0, 1.0]]) / h
    m1 = np.array([[2.0, 1.0], [1.0, 2.0]]) * (h / 6.0)
    e1 = np.array([[0.0, 0.0], [0.0, 1.0]])

    def kron3(z, y, x):
        return np.kron(z, np.kron(y, x))

    return kron3(m1, m1, k1) + kron3(m1, k1, m1) + kron3(k1, m1, m1), kron3(m1, m1, m1), kron3(e1, m1, m1)


class _Mesh:
    """The FEM problem of one case on the GPU: pattern, K, M_c, B_c and what
    the inversion needs."""

    def __init__(self, nx, ny, nz, seed, h=0.05):
        self.h = h
        gen = torch.Generator(DEV).manual_seed(seed)
        self.gen = gen
        f64 = {"dtype": torch.float64, "device": DEV}
        c = C0 * (1.0 + 0.1 * (2.0 * torch.rand(nz, ny, nx, generator=gen, **f64) - 1.0))
        self.c = c.reshape(-1)
        ke, me, bf = _elements(h)
        self.me, self.bf = me, bf

        def pad(t):
            return torch.nn.functional.pad(t, (1, 1, 1, 1, 1, 1))

        one, ic2, top = pad(torch.ones_like(c)), pad(1.0 / (c * c)), torch.zeros_like(c)
        top[-1] = 1.0 / c[-1]
        top = pad(top)
        sh = (nz + 1, ny + 1, nx + 1)
        self.n = n = sh[0] * sh[1] * sh[2]
        kk, jj, ii = torch.meshgrid(*(torch.arange(s, device=DEV) for s in sh), indexing="ij")
        K, M, B = (torch.zeros((27,) + sh, **f64) for _ in range(3))
        exist = torch.zeros((27,) + sh, dtype=torch.bool, device=DEV)
        cols = torch.zeros((27,) + sh, dtype=torch.int64, device=DEV)
        for o, (dz, dy, dx) in enumerate(itertools.product((-1, 0, 1), repeat=3)):
            z, y, x = kk + dz, jj + dy, ii + dx
            # Dirichlet rows and columns (z = 0) leave the pattern
            exist[o] = (z > 0) & (z <= nz) & (y >= 0) & (y <= ny) & (x >= 0) & (x <= nx) & (kk > 0)
            cols[o] = (z * sh[1] + y) * sh[2] + x
            for cz, cy, cx in itertools.product((0, 1), repeat=3):
                az, ay, ax = 1 - cz, 1 - cy, 1 - cx
                bz, by, bx = az + dz, ay + dy, ax + dx
                if min(bz, by, bx) < 0 or max(bz, by, bx) > 1:
                    continue
                a, b = ax + 2 * ay + 4 * az, bx + 2 * by + 4 * bz
                at = (slice(cz, cz + sh[0]), slice(cy, cy + sh[1]), slice(cx, cx + sh[2]))
                K[o] += ke[a, b] * one[at]
                M[o] += me[a, b] * ic2[at]
                if az == 1 and bz == 1:
                    B[o] += bf[a, b] * top[at]
        exist[13] |= kk == 0  # Dirichlet rows are identity rows
        for t, v in ((K, 1.0), (M, 0.0), (B, 0.0)):
            t[13][kk == 0] = v
        exist = exist.reshape(27, n).t()
        self.exist = exist.contiguous()
        self.rowptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
        self.rowptr[1:] = exist.sum(1).cumsum(0)
        self.K, self.M, self.B = (t.reshape(27, n).t()[exist].contiguous() for t in (K, M, B))
        self.colind = cols.reshape(27, n).t()[exist].to(torch.int32).contiguous()
        self.free = (kk > 0).reshape(-1)
        self.xyz = torch.stack([ii, jj, kk], -1).reshape(n, 3)
        self.dims = (nx, ny, nz)

    def omega(self, ppw):
        return 2.0 * math.pi * C0 / (ppw * self.h)

    def values(self, w):
        return torch.complex(self.K - (w * w) * self.M, w * self.B)

    def source(self):
        """A lumped Gaussian point source, sigma = 2 h, somewhere inside."""
        lo = torch.tensor(self.dims, device=DEV, dtype=torch.float64)
        at = lo * (0.25 + 0.5 * torch.rand(3, generator=self.gen, dtype=torch.float64, device=DEV))
        d2 = ((self.xyz - at) ** 2).sum(1)
        return (self.h ** 3 * torch.exp(-d2 / 8.0) * self.free).to(torch.complex128)

    def element_tables(self):
        """CSR slot of every element's node pairs (-1: eliminated) and, per
        slot, its (element, pair) contributions in element order."""
        nx, ny, nz = self.dims
        ez, ey, ex = (t.reshape(-1) for t in torch.meshgrid(*(torch.arange(s, device=DEV) for s in (nz, ny, nx)),
                                                            indexing="ij"))
        loc = [(a & 1, (a >> 1) & 1, a >> 2) for a in range(8)]
        nodes = torch.stack([(ex + ax) + (nx + 1) * ((ey + ay) + (ny + 1) * (ez + az)) for ax, ay, az in loc], 1)
        slot = (self.exist.reshape(-1).cumsum(0) - 1).reshape(self.n, 27)
        emap = torch.empty((nodes.shape[0], 64), dtype=torch.int64, device=DEV)
        for a, b in itertools.product(range(8), repeat=2):
            o = 9 * (loc[b][2] - loc[a][2] + 1) + 3 * (loc[b][1] - loc[a][1] + 1) + loc[b][0] - loc[a][0] + 1
            r = nodes[:, a]
            emap[:, 8 * a + b] = torch.where(self.exist[r, o] & self.free[r], slot[r, o], -1)
        flat = emap.reshape(-1)
        at = torch.nonzero(flat >= 0).reshape(-1)
        s, order = torch.sort(flat[at], stable=True)
        at = at[order]
        pos = torch.arange(s.numel(), device=DEV) - torch.searchsorted(s, s)
        elem = torch.full((self.K.numel(), 8), -1, dtype=torch.int32, device=DEV)
        pair = torch.zeros((self.K.numel(), 8), dtype=torch.uint8, device=DEV)
        elem[s, pos] = (at // 64).to(torch.int32)
        pair[s, pos] = (at % 64).to(torch.uint8)
        return nodes, emap, elem, pair, (ez == nz - 1).to(torch.uint8)


def _vector(n, dtype, gen):
    v = 2.0 * torch.rand(n, 2, generator=gen, dtype=torch.float64, device=DEV) - 1.0
    return torch.view_as_complex(v).to(torch.complex128 if dtype == "c128" else torch.complex64)


def _ragged(case, seed):
    gen = torch.Generator(DEV).manual_seed(seed)
    n, most = case["n"], case["max_row"]
    lens = torch.randint(0, most + 1, (n,), generator=gen, device=DEV)
    lens[torch.rand(n, generator=gen, device=DEV) < 0.1] = 0
    rowptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    rowptr[1:] = lens.cumsum(0)
    # distinct ascending columns: cumulative random gaps, at most n / most each
    gaps = torch.randint(1, max(2, n // most), (n, most), generator=gen, device=DEV)
    keep = torch.arange(most, device=DEV)[None, :] < lens[:, None]
    colind = (gaps.cumsum(1) - 1)[keep].to(torch.int32).contiguous()
    return rowptr, colind, _vector(colind.numel(), case["dtype"], gen), _vector(n, case["dtype"], gen)


_METHODS = {"bicgstab": helm.HELM_BICGSTAB, "tfqmr": helm.HELM_TFQMR, "bicgstabl": helm.HELM_BICGSTABL}
_ELL = 4
_ALPHA, _BETA = 0.6 - 0.8j, 0.3 + 0.4j


def _omegas(case):
    return np.linspace(case["fmin"], case["fmax"], case["freqs"]) * (2.0 * math.pi)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "blas1":
        gen = torch.Generator(DEV).manual_seed(seed)
        x, y = _vector(case["n"], case["dtype"], gen), _vector(case["n"], case["dtype"], gen)
        return {"kind": kind, "x": x, "y": y, "w": torch.empty_like(y),
                "dot": torch.empty(1, dtype=torch.complex128, device=DEV),
                "nrm": torch.empty(1, dtype=torch.float64, device=DEV)}
    if kind == "spmv_ragged":
        rowptr, colind, vals, x = _ragged(case, seed)
        return {"kind": "spmv", "A": helm.CsrMatrix(rowptr, colind, vals), "x": x, "y": torch.empty_like(x)}
    m = _Mesh(case["nx"], case["ny"], case["nz"], seed)
    if kind == "spmv":
        x = _vector(m.n, case["dtype"], m.gen)
        vals = m.values(m.omega(case["ppw"])).to(x.dtype)
        return {"kind": kind, "A": helm.CsrMatrix(m.rowptr, m.colind, vals), "x": x, "y": torch.empty_like(x)}
    b = m.source()
    if kind == "sweep":
        return {"kind": kind, "S": helm.Sweep(m.rowptr, m.colind, m.K, m.M, m.B), "b": b, "w": _omegas(case),
                "X": torch.zeros((m.n, case["freqs"]), dtype=torch.complex128, device=DEV),
                "opts": {"tol": case["tol"], "maxit": 100000}}
    w = m.omega(case["ppw"])
    if kind == "inversion":
        _, emap, elem, pair, top = m.element_tables()
        fem = hgrad.HelmholtzFEM(m.rowptr, m.colind, m.K, elem, pair, emap, m.me, m.bf, top, w, DEV)
        rec, d = _receivers(m)
        return {"kind": kind, "fem": fem, "c": m.c.requires_grad_(True), "b": b.requires_grad_(True), "rec": rec, "d": d,
                "opts": helm.default_opts(tol=case["tol"], maxit=100000)}
    A = helm.CsrMatrix(m.rowptr, m.colind, m.values(w))
    opts = {"tol": case["tol"], "maxit": 200000}
    if kind == "mixed":
        opts["precision"] = helm.HELM_PREC_MIXED
    else:
        opts.update(method=_METHODS[case["method"]], ell=_ELL)
    return {"kind": kind, "A": A, "b": b, "x": torch.empty_like(b), "opts": opts}


def _receivers(m):
    at = torch.nonzero(m.free).reshape(-1)
    rec = at[torch.randperm(at.numel(), generator=m.gen, device=DEV)[:64]]
    return rec, 1e-3 * _vector(64, "c128", m.gen)


def run(state):
    kind = state["kind"]
    if kind == "blas1":
        x, y, w = state["x"], state["y"], state["w"]
        helm.helm_axpby(1.0, x, 0.0, w)      # w = x
        helm.helm_axpby(_ALPHA, y, 1.0, w)   # w = alpha y + w
        helm.helm_axpby(0.0, x, _BETA, w)    # w = beta w
        helm.helm_dot(w, y, state["dot"])
        helm.helm_nrm2(w, state["nrm"])
        return {"w": w, "dot": state["dot"], "nrm": state["nrm"]}
    if kind == "spmv":
        return state["A"].matvec(state["x"], state["y"])
    if kind == "sweep":
        X, _ = state["S"].solve(state["w"], state["b"], state["X"], **state["opts"])
        return {"X": X}
    if kind == "inversion":
        u = hgrad.solve_sound_speed(state["c"], state["b"], state["fem"], state["opts"])
        e = u[state["rec"]] - state["d"]
        loss = (e.real ** 2 + e.imag ** 2).sum()
        gc, gb = torch.autograd.grad(loss, (state["c"], state["b"]))
        return {"u": u.detach(), "grad_c": gc, "grad_b": gb}
    x, _ = helm.solve(state["A"], state["b"], state["x"], **state["opts"])
    return {"x": x}


def _sizes(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    return (nx + 1) * (ny + 1) * (nz + 1), (3 * nx + 1) * (3 * ny + 1) * (3 * nz - 2) + (nx + 1) * (ny + 1)


def work(case):
    kind = case["kind"]
    if kind == "blas1":
        z = 16 if case["dtype"] == "c128" else 8
        # copy 2, axpy 3, scale 2, dot 2 and norm 1 vectors; 8 + 6 + 8 + 4 real operations per element
        return {"bytes": 10.0 * z * case["n"], "flops": 26.0 * case["n"]}
    if kind == "spmv_ragged":
        z, n = 16 if case["dtype"] == "c128" else 8, case["n"]
        nnz = 0.45 * case["max_row"] * n
        return {"bytes": (z + 4) * nnz + (2 * z + 4) * n, "flops": 8.0 * nnz}
    n, nnz = _sizes(case)
    if kind == "spmv":
        z = 16 if case["dtype"] == "c128" else 8
        return {"bytes": (z + 4.0) * nnz + (2 * z + 4) * n, "flops": 8.0 * nnz}
    # a whole solve: some products with A, and the vectors of an iteration
    if kind == "sweep":
        # K, M and B once for all frequencies
        f = case["freqs"]
        return {"bytes": 4000.0 * (28 * nnz + 32 * n * f), "flops": 4000.0 * f * (6 * nnz + 40 * n)}
    z = 8 if kind == "mixed" else 16
    return {"bytes": 4000.0 * ((z + 4) * nnz + 4 * z * n), "flops": 4000.0 * (4 * nnz + 46 * n)}


# ---------------------------------------------------------------- 64 bits, in plain torch

class _Csr:
    def __init__(self, rowptr, colind, vals):
        self.n = rowptr.numel() - 1
        self.rows = torch.repeat_interleave(torch.arange(self.n, device=DEV), (rowptr[1:] - rowptr[:-1]).long())
        self.cols, self.vals = colind.long(), vals

    def __matmul__(self, x):
        y = torch.zeros(self.n, dtype=torch.complex128, device=DEV)
        return y.index_add_(0, self.rows, self.vals * x[self.cols])


def _dot(a, b):
    return (a.conj() * b).sum(0)


def _bicgstabl(A, b, tol, ell=4, cycles=20000):
    """Sleijpen & Fokkema 1993, from x = 0."""
    x, rt = torch.zeros_like(b), b.clone()
    R, U = [b.clone()], [torch.zeros_like(b)]
    one = torch.ones((), dtype=torch.complex128, device=DEV)
    rho0, alpha, omega = one, 0 * one, one
    stop = tol * float(torch.linalg.vector_norm(b))
    for _ in range(cycles):
        rho0 = -omega * rho0
        for j in range(ell):
            rho1 = _dot(rt, R[j])
            beta = alpha * rho1 / rho0
            rho0 = rho1
            U = [R[i] - beta * U[i] for i in range(j + 1)]
            U.append(A @ U[j])
            alpha = rho0 / _dot(rt, U[j + 1])
            R = [R[i] - alpha * U[i + 1] for i in range(j + 1)]
            R.append(A @ R[j])
            x = x + alpha * U[0]
        Z = torch.stack(R[1:], 1)
        Q, T = torch.linalg.qr(Z)
        g = torch.linalg.solve_triangular(T, (Q.mH @ R[0])[:, None], upper=True)[:, 0]
        omega = g[ell - 1]
        x = x + torch.stack(R[:ell], 1) @ g
        R = [R[0] - Z @ g]
        U = [U[0] - torch.stack(U[1:], 1) @ g]
        if float(torch.linalg.vector_norm(R[0])) <= stop:
            break
    return x


def _solve(A, b):
    """A x = b: dense when it fits, else iterated, and refined on its residual."""
    if A.n <= 8000:
        D = torch.zeros((A.n, A.n), dtype=torch.complex128, device=DEV)
        D[A.rows, A.cols] = A.vals
        return torch.linalg.solve(D, b)
    x = _bicgstabl(A, b, 1e-8)
    for _ in range(2):
        x = x + _bicgstabl(A, b - A @ x, 1e-4)
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "blas1":
        gen = torch.Generator(DEV).manual_seed(seed)
        x, y = (_vector(case["n"], case["dtype"], gen).to(torch.complex128) for _ in range(2))
        w = _BETA * (x + _ALPHA * y)
        return {"w": w, "dot": _dot(w, y).reshape(1), "nrm": torch.linalg.vector_norm(w).reshape(1)}
    if kind == "spmv_ragged":
        rowptr, colind, vals, x = _ragged(case, seed)
        return _Csr(rowptr, colind, vals.to(torch.complex128)) @ x.to(torch.complex128)
    m = _Mesh(case["nx"], case["ny"], case["nz"], seed)
    if kind == "spmv":
        x = _vector(m.n, case["dtype"], m.gen)
        vals = m.values(m.omega(case["ppw"])).to(x.dtype)
        return _Csr(m.rowptr, m.colind, vals.to(torch.complex128)) @ x.to(torch.complex128)
    b = m.source()
    if kind == "sweep":
        if case["freqs"] * m.n > 200_000:
            return None
        As = (_Csr(m.rowptr, m.colind, m.values(w)) for w in _omegas(case))
        return {"X": torch.stack([_solve(A, b) for A in As], 1)}
    w = m.omega(case["ppw"])
    A = _Csr(m.rowptr, m.colind, m.values(w))
    u = _solve(A, b)
    if kind != "inversion":
        return {"x": u}
    nodes, emap, _, _, top = m.element_tables()
    rec, d = _receivers(m)
    rhs = torch.zeros_like(b)
    rhs[rec] = (u[rec] - d).conj()
    mu = _solve(A, rhs)  # A is its own transpose
    me, bf = (torch.as_tensor(t, device=DEV).reshape(1, 64) for t in (m.me, m.bf))
    G = -(mu[nodes][:, :, None] * u[nodes][:, None, :]).reshape(-1, 64) * (emap >= 0)
    c = m.c[:, None]
    dA = torch.complex((2.0 * w * w / c ** 3) * me, -(w / c ** 2) * bf * top[:, None])
    return {"u": u, "grad_c": 2.0 * (G * dA).sum(1).real, "grad_b": 2.0 * mu.conj()}
