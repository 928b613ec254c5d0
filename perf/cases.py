"""Timed workloads of the framework's public entry points.

Each case is one call (or the short sequence of calls) that a program using
the Python binding makes on a problem it has set up: a product with A, a
preconditioner application, a whole solve, a batched solve, the set-up of a
patch. The problems are the deformed unit cube (3D) and the identity square
(2D) with N(0, 1) vectors; the deformation and the vectors come from the seed.
"""
import math

import numpy as np
import torch

from paper_1602_01636_gb300 import igafd

TOL = 1e-8          # relative residual of every solve
AMP = 0.05          # amplitude bound of the cube's deformation
ADI_STEPS = 8       # ADI iterations per application (reaches about 0.1 at n = 128)


def listed():
    return [
        # the smallest solve: a 2D patch whose preconditioner equals A (one iteration); latency
        {"name": "solve_2d_64", "op": "solve", "n1": 64, "n2": 64, "n3": 0, "p": 3, "dtype": "fp64"},
        # the product with A inside every iteration, at the benchmark's size
        {"name": "apply_a_128_p3", "op": "apply_a", "n1": 128, "n2": 128, "n3": 128, "p": 3, "half": False},
        # the same on a patch of uneven directions and a higher degree
        {"name": "apply_a_ragged_p4", "op": "apply_a", "n1": 61, "n2": 90, "n3": 47, "p": 4, "half": False},
        # the paper's preconditioner in its own arithmetic (the binding's default dtype)
        {"name": "prec_fp64_128", "op": "prec", "n1": 128, "n2": 128, "n3": 128, "p": 3, "dtype": "fp64"},
        {"name": "prec_fp64_ragged", "op": "prec", "n1": 95, "n2": 61, "n3": 77, "p": 2, "dtype": "fp64"},
        # the mixed-precision preconditioner at the benchmark's size, and on uneven directions
        {"name": "prec_tf32_128", "op": "prec", "n1": 128, "n2": 128, "n3": 128, "p": 3, "dtype": "tf32"},
        {"name": "prec_bf16_ragged", "op": "prec", "n1": 70, "n2": 45, "n3": 93, "p": 3, "dtype": "bf16"},
        # the benchmark's step: set-up of P and the mixed-precision solve
        {"name": "solve_tf32_128", "op": "solve", "n1": 128, "n2": 128, "n3": 128, "p": 3, "dtype": "tf32"},
        # the all-FP64 solve with the binding's defaults
        {"name": "solve_fp64_64", "op": "solve", "n1": 64, "n2": 64, "n3": 64, "p": 3, "dtype": "fp64"},
        # many problems of uneven sizes and degrees at once
        {"name": "batch_8", "op": "batch", "count": 8, "lo": 32, "hi": 64, "dtype": "bf16"},
        # a new geometry: patch set-up (assembly of A, set-up of P), its load vector, A handed out
        {"name": "setup_56_p3", "op": "setup", "n1": 56, "n2": 56, "n3": 56, "p": 3, "half": False},
        # the paper's other preconditioner
        {"name": "adi_fp64_96", "op": "adi", "n1": 96, "n2": 96, "n3": 96, "p": 3, "dtype": "fp64"},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["solve", "solve_2d", "apply_a", "prec", "prec", "prec_2d", "batch", "setup", "adi"])
    dtypes = ["fp64", "fp64", "tf32", "bf16", "fp32", "fp16"]
    if op == "batch":
        return {"op": op, "count": rng.randint(2, 8), "lo": rng.randint(20, 32), "hi": rng.randint(40, 64),
                "dtype": rng.choice(["bf16", "tf32", "fp64"])}
    if op in ("solve_2d", "prec_2d"):
        return {"op": op[:-3], "n1": size(16, 160), "n2": size(16, 160), "n3": 0, "p": rng.randint(1, 5),
                "dtype": rng.choice(dtypes)}
    most = {"solve": 100, "apply_a": 112, "prec": 160, "setup": 56, "adi": 96}[op]
    case = {"op": op, "n1": size(12, most), "n2": size(12, most), "n3": size(12, most), "p": rng.randint(2, 4)}
    if op in ("solve", "prec"):
        case["dtype"] = rng.choice(dtypes)
    elif op == "adi":
        case["dtype"] = rng.choice(["fp64", "fp32"])
    else:
        case["half"] = rng.random() < 0.25
    return case


# ---- the problem's inputs ------------------------------------------------------
def sizes(case):
    return [case["n1"], case["n2"]] + ([case["n3"]] if case["n3"] else [])


def open_knots(n, p):
    """Uniform open knots whose degree-p space has n functions that vanish at both ends."""
    return np.concatenate([np.zeros(p), np.linspace(0.0, 1.0, n - p + 3), np.ones(p)])


def control_net(knots, p, amplitudes):
    """Greville points [c][i_d]..[i_1] (the identity map), in 3D displaced by
    sum_k a_k sin(k pi x) sin(k pi y) sin(k pi z) (1, 1, 1)."""
    g = [np.array([k[i + 1:i + p + 1].mean() for i in range(len(k) - p - 1)]) for k in knots]
    net = np.stack(np.meshgrid(*g[::-1], indexing="ij")[::-1])
    if len(g) == 3:
        net = net + sum(a * np.prod(np.sin(k * np.pi * net), axis=0) for k, a in enumerate(amplitudes, 1))
    return np.ascontiguousarray(net)


def geometry(n, p, rng):
    knots = [open_knots(v, p) for v in n]
    return knots, control_net(knots, p, rng.uniform(-AMP, AMP, size=3))


def vector(N, rng):
    return torch.from_numpy(rng.standard_normal(N)).cuda()


def batch_problems(case, seed):
    """(n, p) of every problem (fixed by the case), geometry and right-hand side (from the seed)."""
    shape = np.random.Generator(np.random.PCG64([case["count"], case["lo"], case["hi"]]))
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for _ in range(case["count"]):
        n, p = [int(v) for v in shape.integers(case["lo"], case["hi"] + 1, size=3)], int(shape.integers(2, 5))
        knots, net = geometry(n, p, rng)
        out.append((knots, p, net, rng.standard_normal(int(np.prod(n)))))
    return out


def adi_parameters(n):
    """Geometrically spaced positive parameters over the spectra's range (pi^2 to about 10 n^2)."""
    top = 10.0 * max(n) ** 2
    return np.pi ** 2 * (top / np.pi ** 2) ** (np.arange(ADI_STEPS) / (ADI_STEPS - 1.0))


def prepare(case, seed):
    op = case["op"]
    if op == "batch":
        probs = batch_problems(case, seed)
        patches = [igafd.Patch(kn, p, net) for kn, p, net, _ in probs]
        return {"op": op, "batch": igafd.Batch(patches, tol=TOL, dtype=case["dtype"], groups=0),
                "b": [torch.from_numpy(b).cuda() for _, _, _, b in probs]}
    rng = np.random.Generator(np.random.PCG64(seed))
    knots, net = geometry(sizes(case), case["p"], rng)
    if op == "setup":
        return {"op": op, "knots": knots, "p": case["p"], "net": net, "half": case["half"]}
    stencil = op in ("apply_a", "solve")
    patch = igafd.Patch(knots, case["p"], net, stencil=stencil, half_stencil=stencil and case.get("half", False))
    if op == "adi":
        patch.adi_setup(adi_parameters(sizes(case)), dtype=case["dtype"])
    return {"op": op, "patch": patch, "v": vector(patch.N, rng), "dtype": case.get("dtype")}


def run(state):
    op = state["op"]
    if op == "apply_a":
        return state["patch"].apply_A(state["v"])
    if op == "prec":
        return state["patch"].apply_prec(state["v"], dtype=state["dtype"])
    if op == "adi":
        return state["patch"].apply_prec_adi(state["v"])
    if op == "solve":
        # a time to solution includes the set-up of P, as the paper's timings do
        state["patch"].setup_prec()
        return state["patch"].pcg(state["v"], tol=TOL, dtype=state["dtype"])[0]
    if op == "batch":
        return state["batch"].solve(state["b"])[0]
    patch = igafd.Patch(state["knots"], state["p"], state["net"], half_stencil=state["half"])
    out = {"b": patch.load_rhs_sine(), "A": patch.stencil()}
    patch.close()
    return out


# ---- what a pass cannot do without --------------------------------------------
def couplings(n, p):
    """Nonzero entries of A: per direction n (2p + 1) minus the couplings that leave the box."""
    out = 1
    for v in n:
        out *= sum(max(0, v - abs(d)) for d in range(-p, p + 1))
    return out


def solve_work(n, p, iterations):
    """Per iteration A read once, a product with A, a preconditioner application, the vector updates."""
    N, nnz = math.prod(n), couplings(n, p)
    return iterations * (8 * nnz + 72 * N), iterations * (2 * nnz + 4 * N * sum(n) + 12 * N)


def work(case):
    op = case["op"]
    if op == "batch":
        per = [solve_work([len(k) - p - 3 for k in kn], p, 16) for kn, p, _, _ in batch_problems(case, 0)]
        return {"bytes": sum(b for b, _ in per), "flops": sum(f for _, f in per)}
    n, p = sizes(case), case["p"]
    N, nnz = math.prod(n), couplings(n, p)
    if op == "apply_a":
        stored = (nnz + N) / 2 if case["half"] else nnz
        return {"bytes": 8 * stored + 16 * N, "flops": 2 * nnz}
    if op == "prec":
        return {"bytes": 16 * N, "flops": 4 * N * sum(n)}
    if op == "adi":
        return {"bytes": 16 * N, "flops": ADI_STEPS * (36 * p + 29) * N}
    if op == "solve":
        # iterations to the tolerance: one on the identity map, about 16 on the deformed cube
        b, f = solve_work(n, p, 16 if len(n) == 3 else 1)
        return {"bytes": b, "flops": f}
    # set-up: A written once and handed out once; assembly contracts Q's three-by-three terms over the
    # quadrature points one direction after the other, for the couplings of one triangle
    q, w = p + 1, 2 * p + 1
    pairs = q * q * q          # (coupling, point) pairs per function and direction
    stored = (nnz + N) / 2 if case["half"] else nnz
    return {"bytes": 8 * (stored + 2 * nnz), "flops": N * (9 * pairs * q * q + 9 * w * pairs * q + 4 * w * w * pairs)}


# ---- 64-bit values --------------------------------------------------------------
def basis(knots, p, z):
    """Values and first derivatives [point][function] of every degree-p B-spline at interior points."""
    N = ((knots[None, :-1] <= z[:, None]) & (z[:, None] < knots[None, 1:])).astype(float)
    low = N
    for q in range(1, p + 1):
        low = N
        a, b = knots[q:-1] - knots[:-q - 1], knots[q + 1:] - knots[1:-q]
        ra = np.divide(1.0, a, out=np.zeros_like(a), where=a > 0)
        rb = np.divide(1.0, b, out=np.zeros_like(b), where=b > 0)
        N = (z[:, None] - knots[None, :-q - 1]) * ra * low[:, :-1] + (knots[None, q + 1:] - z[:, None]) * rb * low[:, 1:]
    return N, p * (ra * low[:, :-1] - rb * low[:, 1:])


class Exact:
    """The problem in plain torch, FP64: basis tables at the (p + 1)-point Gauss points, Q there."""

    def __init__(self, knots, p, net=None):
        self.d, self.p = len(knots), p
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        xg, wg = np.polynomial.legendre.leggauss(p + 1)
        self.V, self.D, self.w, self.pencil = [], [], [], []
        for k in knots:
            e = np.unique(k)
            z = (0.5 * (e[:-1] + e[1:])[:, None] + 0.5 * np.diff(e)[:, None] * xg).ravel()
            w = (0.5 * np.diff(e)[:, None] * wg).ravel()
            V, D = basis(k, p, z)
            self.w.append(torch.from_numpy(w).to(self.dev))
            self.V.append(torch.from_numpy(V).to(self.dev))
            self.D.append(torch.from_numpy(D).to(self.dev))
            v, g = V[:, 1:-1], D[:, 1:-1]
            self.pencil.append((g.T @ (w[:, None] * g), v.T @ (w[:, None] * v)))
        self.n = [t.shape[1] - 2 for t in self.V]
        if net is not None:
            self.coefficient(torch.from_numpy(net).to(self.dev))

    def along(self, T, x, k):
        """Contract direction k (0 the fastest, the last axis) of x with the table T[out][in]."""
        ax = self.d - 1 - k
        return torch.movedim(torch.tensordot(T, x, dims=([1], [ax])), 0, ax)

    def tensor(self, tables, x):
        for k, T in enumerate(tables):
            x = self.along(T, x, k)
        return x

    def coefficient(self, net):
        d = self.d
        self.x = [self.tensor(self.V, net[c]) for c in range(d)]
        J = [[self.tensor([self.D[k] if k == j else self.V[k] for k in range(d)], net[c]) for j in range(d)]
             for c in range(d)]
        wt = self.w[0]
        for k in range(1, d):
            wt = self.w[k].reshape([-1] + [1] * k) * wt
        if d == 2:
            adj = [[J[1][1], -J[0][1]], [-J[1][0], J[0][0]]]
            det = J[0][0] * J[1][1] - J[0][1] * J[1][0]
        else:
            def cof(r, c):
                (a, b), (e, f) = [[i for i in range(3) if i != q] for q in (r, c)]
                return (-1) ** (r + c) * (J[a][e] * J[b][f] - J[a][f] * J[b][e])
            adj = [[cof(c, r) for c in range(3)] for r in range(3)]
            det = sum(J[0][c] * adj[c][0] for c in range(3))
        del J
        self.wdet = wt * det.abs()
        # Q = |det| J^-1 J^-T with J^-1 = adj / det
        self.Q = {(r, s): (wt / det.abs()) * sum(adj[r][i] * adj[s][i] for i in range(d))
                  for r in range(d) for s in range(r, d)}

    def inner(self, r):
        """Tables of the kept functions, the derivative in direction r."""
        return [(self.D[k] if k == r else self.V[k])[:, 1:-1] for k in range(self.d)]

    def A(self, x):
        x = x.reshape(self.n[::-1])
        g = [self.tensor(self.inner(s), x) for s in range(self.d)]
        y = 0.0
        for r in range(self.d):
            f = sum(self.Q[min(r, s), max(r, s)] * g[s] for s in range(self.d))
            y = y + self.tensor([T.T for T in self.inner(r)], f)
        return y.reshape(-1)

    def eigen(self):
        """Generalised eigenvectors per direction and the eigenvalues, shaped to their direction's axis."""
        U, lam = [], []
        for k, (K, M) in enumerate(self.pencil):
            Li = np.linalg.inv(np.linalg.cholesky(M))
            S = Li @ K @ Li.T
            D, W = np.linalg.eigh(0.5 * (S + S.T))
            U.append(torch.from_numpy(Li.T @ W).to(self.dev))
            lam.append(torch.from_numpy(D).to(self.dev).reshape([-1] + [1] * k))
        return U, lam

    def P(self, r, omega=None):
        """P^-1 r, or with ADI parameters the result of that many ADI steps from zero (the error of a
        step is diagonal in the generalised eigenvectors)."""
        if not hasattr(self, "spectrum"):
            self.spectrum = self.eigen()
        U, lam = self.spectrum
        t = self.tensor([u.T for u in U], r.reshape(self.n[::-1])) / sum(lam)
        if omega is not None:
            err = 1.0
            for w in omega:
                err = err * (1.0 - 2.0 * w * w * sum(lam) / ((w + lam[0]) * (w + lam[1]) * (w + lam[2])))
            t = t * (1.0 - err)
        return self.tensor(U, t).reshape(-1)

    def solve(self, b, tol=1e-12, most=200):
        x, r = torch.zeros_like(b), b.clone()
        z = self.P(r)
        p, rz = z.clone(), torch.dot(r, z)
        for _ in range(most):
            q = self.A(p)
            a = rz / torch.dot(p, q)
            x, r = x + a * p, r - a * q
            if float(r.norm()) <= tol * float(b.norm()):
                break
            z = self.P(r)
            rz, old = torch.dot(r, z), rz
            p = z + (rz / old) * p
        return x

    def load(self):
        """The load of u = prod_k sin(pi x_k): f = d pi^2 u."""
        f = self.d * np.pi ** 2 * self.wdet
        for x in self.x:
            f = f * torch.sin(np.pi * x)
        return self.tensor([T.T for T in self.inner(None)], f).reshape(-1)

    def stencil(self):
        """A as [(2p + 1)^3][N]: entry [o][row] = A[row, row + delta], zero outside the box."""
        p, n = self.p, self.n
        W = 2 * p + 1
        out = torch.zeros([W, W, W] + n[::-1], dtype=torch.float64, device=self.dev)

        def pair(k, a, b, dl):
            """[i][point]: table a at i times table b at i + dl (zero where i + dl leaves the box)."""
            lo, hi = max(0, -dl), n[k] - max(0, dl)
            T = torch.zeros(n[k], a.shape[0], dtype=torch.float64, device=self.dev)
            if hi > lo:
                T[lo:hi] = a[:, lo:hi].T * b[:, lo + dl:hi + dl].T
            return T

        for r in range(3):
            for s in range(3):
                fr, fs, Q = self.inner(r), self.inner(s), self.Q[min(r, s), max(r, s)]
                for d1 in range(W):
                    q1 = self.along(pair(0, fr[0], fs[0], d1 - p), Q, 0)
                    for d2 in range(W):
                        q2 = self.along(pair(1, fr[1], fs[1], d2 - p), q1, 1)
                        for d3 in range(W):
                            out[d3, d2, d1] += self.along(pair(2, fr[2], fs[2], d3 - p), q2, 2)
        return out.reshape(W ** 3, -1)


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        out = []
        for knots, p, net, b in batch_problems(case, seed):
            e = Exact(knots, p, net)
            out.append(e.solve(torch.from_numpy(b).to(e.dev)))
        return out
    rng = np.random.Generator(np.random.PCG64(seed))
    knots, net = geometry(sizes(case), case["p"], rng)
    e = Exact(knots, case["p"], net if op in ("apply_a", "solve", "setup") else None)
    if op == "setup":
        return {"b": e.load(), "A": e.stencil()}
    v = torch.from_numpy(rng.standard_normal(math.prod(e.n))).to(e.dev)
    if op == "apply_a":
        return e.A(v)
    if op == "prec":
        return e.P(v)
    if op == "adi":
        return e.P(v, adi_parameters(e.n))
    return e.solve(v)
