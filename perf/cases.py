"""Performance cases of the Karhunen-Loeve library: what a program that uses it has it do.

Each case is one call, or one short fixed sequence of calls, of the C ABI
(include/kl.h) through its Python binding, on the meshes, kernels and block
widths of this repository's own workloads (kl_inputs, the accuracy studies of
bench.py, the parity tests):

  apply    Y = A X or A' X (kl_apply_A, kl_apply_Aprime): the matrix-free
           operator for a program that has its own outer iteration
  zinv     Y = Z^-1 X (kl_apply_Zinv)
  pairs    the pairwise product alone on caller-given points
           (kl_pairwise_noalloc)
  sample   realisations of the truncated expansion (kl_sample)
  eigs     the M leading eigenpairs (kl_eigs)

Blocks keep the type their arithmetic has: FP64 handles give FP64 results; the
results of the reduced-precision handles (FP32 kernel values) are kept in FP32,
which is what they are good for.

exact() evaluates the same discrete operators in 64 bits with plain
numpy/torch: textbook B-splines, the Kronecker factors and dense kernel rows.
"""
import math

import numpy as np
import torch

import paper_2101_00629_gb300 as kl

SQRT_HALF = math.sqrt(0.5)


def listed():
    return [
        # smallest call: one vector on the 216-dof cube of the parity workload,
        # an outer iteration of the caller's own in FP64; launches count
        dict(name="apply_f64_cube4_k1", op="apply", form="A", geometry="cube", p=2, e1=4, e2=4, e3=4, kernel="gauss",
             L=0.5, method="galerkin", precision="fp64", k=1),
        # the half cylinder of the h-refinement study (mesh 3 of 5), FP64:
        # the library's default precision, one block of the eigensolver
        dict(name="apply_f64_halfcyl_galerkin", op="apply", form="Aprime", geometry="half_annulus", p=2, e1=32, e2=2,
             e3=18, kernel="exp", L=5.0, method="galerkin", precision="fp64", k=8),
        # its k-refinement study at degree 6 (Gaussian kernel), collocation:
        # many quadrature points, the smooth kernel needs FP64
        dict(name="apply_f64_halfcyl_colloc_p6", op="apply", form="Aprime", geometry="half_annulus", p=6, e1=32, e2=1,
             e3=8, kernel="gauss", L=5.0, method="collocation", precision="fp64", k=8),
        # FP32 handle, ragged block width, degree 3, Matern kernel, weights
        # that are not a tensor product
        dict(name="apply_f32_projective_k5", op="apply", form="A", geometry="projective_cube", p=3, e1=13, e2=11, e3=9,
             kernel="matern32", L=0.7, method="collocation", precision="fp32", k=5),
        # the benchmark workload's Galerkin operator, split BF16
        dict(name="apply_bf16_cube16_galerkin", op="apply", form="Aprime", geometry="cube", p=2, e1=16, e2=16, e3=16,
             kernel="exp_sep", L=1.0, method="galerkin", precision="bf16", k=8),
        # the degree-3 annulus workload's collocation operator, split BF16
        dict(name="apply_bf16_annulus_colloc", op="apply", form="Aprime", geometry="annulus", p=3, e1=32, e2=32, e3=16,
             kernel="gauss", L=0.5, method="collocation", precision="bf16", k=16),
        # the largest: the 64x32x16 annulus workload's Galerkin operator at its
        # block width
        dict(name="apply_bf16_annulus64_galerkin", op="apply", form="Aprime", geometry="annulus", p=2, e1=64, e2=32,
             e3=16, kernel="exp", L=1.0, method="galerkin", precision="bf16", k=32),
        # kernel matrix products on scattered points, odd sizes, few columns
        dict(name="pairs_f64_scattered", op="pairs", T=5003, S=20011, kernel="matern32", L=0.4, k=3),
        # mass-matrix solves on the large annulus mesh (projections of M = 32
        # fields onto the trial space)
        dict(name="zinv_annulus64", op="zinv", geometry="annulus", p=2, e1=64, e2=32, e3=16, kernel="exp", L=1.0,
             method="galerkin", precision="fp64", k=32),
        # 1024 realisations of the 20-mode expansion on the benchmark mesh
        dict(name="sample_cube16", op="sample", geometry="cube", p=2, e1=16, e2=16, e3=16, kernel="exp_sep", L=1.0,
             method="galerkin", precision="bf16", M=20, ns=1024),
        # a whole FP64 solve with vectors: no symmetry, so that every pair is
        # determined
        dict(name="eigs_f64_projective", op="eigs", geometry="projective_cube", p=2, e1=8, e2=7, e3=6, kernel="exp",
             L=0.9, method="galerkin", precision="fp64", k=8, M=8, vectors=True),
        # the benchmark workload's Galerkin solve, split BF16: values only (the
        # cube's repeated eigenvalues leave their vectors undetermined)
        dict(name="eigs_bf16_cube16", op="eigs", geometry="cube", p=2, e1=16, e2=16, e3=16, kernel="exp_sep", L=1.0,
             method="galerkin", precision="bf16", k=8, M=20, vectors=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# pairs (targets x sources) a drawn application may have, by precision: each
# stays below the largest listed case
MOST_PAIRS = {"fp64": 3e8, "fp32": 2e9, "bf16": 2e10, "tf32": 8e9}


def draw(rng):
    op = rng.choice(["apply", "apply", "apply", "pairs", "zinv", "sample", "eigs"])
    kernel = rng.choice(["gauss", "exp_sep", "exp", "matern32"])
    L = round(_log(rng, 0.1, 2.0), 4)
    if op == "pairs":
        return dict(op=op, T=int(_log(rng, 33, 30000)), S=int(_log(rng, 33, 30000)), kernel=kernel, L=L,
                    k=int(_log(rng, 1, 17)))
    while True:
        geometry = rng.choice(["cube", "annulus", "half_annulus", "projective_cube"])
        e = [max(1, int(_log(rng, 2, 28))) for _ in range(3)]
        if geometry == "half_annulus":
            e[0] += e[0] % 2
        c = dict(op=op, geometry=geometry, p=rng.choice([2, 2, 3, 4]), e1=e[0], e2=e[1], e3=e[2], kernel=kernel, L=L,
                 method=rng.choice(["galerkin", "galerkin", "collocation", "collocation", "galerkin_std"]),
                 precision=rng.choice(["fp64", "fp64", "fp32", "bf16", "bf16", "tf32"]))
        if op == "sample":
            c.update(M=rng.randint(5, 40), ns=int(_log(rng, 16, 512)), method=rng.choice(["galerkin", "collocation"]))
            if e[0] * e[1] * e[2] * (c["p"] + 1) ** 3 * c["ns"] <= 5e7:
                return c
            continue
        if op == "zinv":
            c.update(k=int(_log(rng, 1, 65)), precision="fp64")
            return c
        c["k"] = int(_log(rng, 1, 33)) if op == "apply" else 8
        N, S, T = _sizes(c)
        if op == "apply":
            c["form"] = rng.choice(["A", "Aprime"])
            if S * T <= MOST_PAIRS[c["precision"]] * (1.0 if c["k"] <= 8 else 8.0 / c["k"]):
                return c
            continue
        # whole solves: bases of a few hundred dofs and more, correlation
        # lengths the split operands resolve
        c.update(M=rng.randint(4, 12), vectors=False, method=rng.choice(["galerkin", "collocation"]),
                 precision=rng.choice(["fp64", "bf16"]))
        c["L"] = round(_log(rng, 0.4 if c["precision"] == "fp64" else 0.8, 2.0), 4)
        N, S, T = _sizes(c)
        if N >= 300 and S * T <= (2e7 if c["precision"] == "fp64" else 4e8):
            return c


# ---------------------------------------------------------------------------
# The program's side: handle, inputs, calls
# ---------------------------------------------------------------------------

GEO = {"cube": (1.0, 2.0, 1.0), "annulus": (1.0, 2.0, 1.0), "projective_cube": (0.5, 0.25, -0.2)}


def _geo(case):
    # half cylinder: the shell of the accuracy studies at L = 5, else the unit
    # radius one
    if case["geometry"] == "half_annulus":
        return (27.5, 30.5, 23.0) if case["L"] > 2.0 else (1.0, 2.0, 1.0)
    return GEO[case["geometry"]]


def _length(case, seed):
    """Correlation length: of a solve it is part of the input."""
    if case["op"] != "eigs":
        return case["L"]
    return case["L"] * (1.0 + 0.02 * float(np.random.default_rng(seed).uniform(-1.0, 1.0)))


class Handle:
    def __init__(self, case, seed):
        p = kl.params(geometry=case["geometry"], degree=case["p"], elems=(case["e1"], case["e2"], case["e3"]),
                      kernel=case["kernel"], sigma=1.0, L=_length(case, seed), method=case["method"],
                      precision=case["precision"], block_k=min(64, case.get("k", 8)), geo=_geo(case),
                      seed=2101 + seed % 1000)
        self.h = kl.kl_create(p, torch.cuda.current_stream())
        self.N, self.S, self.T = kl.kl_dims(self.h)

    def __del__(self):
        if getattr(self, "h", None):
            kl.kl_destroy(self.h)


def _normal(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _modes(case, seed):
    """Variances and coefficient vectors of smooth modes (products of cosines
    of the three directions), and the standard normal variables."""
    r = np.random.default_rng(seed)
    n = [case[f"e{d}"] + case["p"] for d in (1, 2, 3)]
    if case["geometry"] == "half_annulus":
        n[0] += case["p"] - 1
    lam = 1.0 / (1.0 + np.arange(case["M"])) ** 2
    V = np.empty((case["M"], n[0] * n[1] * n[2]))
    for m in range(case["M"]):
        f = [np.cos(math.pi * r.integers(0, 5) * np.linspace(0, 1, n[d]) + 0.3 * r.uniform()) for d in range(3)]
        V[m] = np.einsum("k,j,i->kji", f[2], f[1], f[0]).reshape(-1)
    return lam, torch.from_numpy(V).cuda(), _normal(seed, case["ns"], case["M"])


def _points(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.rand(3, case[n], generator=g, device="cuda", dtype=torch.float64) for n in ("T", "S")]


def prepare(case, seed):
    s = {"case": case}
    if case["op"] == "pairs":
        s["tgt"], s["src"] = _points(case, seed)
        s["X"] = _normal(seed + 1, case["k"], case["S"])
        s["Y"] = torch.empty(case["k"], case["T"], device="cuda", dtype=torch.float64)
        return s
    s["handle"] = h = Handle(case, seed)
    if case["op"] in ("apply", "zinv"):
        s["X"] = _normal(seed, case["k"], h.N)
        s["Y"] = torch.empty_like(s["X"])
    elif case["op"] == "sample":
        s["lam"], s["V"], s["xi"] = _modes(case, seed)
        s["out"] = torch.empty(case["ns"], kl.kl_sample_size(h.h), device="cuda", dtype=torch.float64)
    else:
        s["lam"] = np.zeros(case["M"])
        s["V"] = torch.empty(case["M"], h.N, device="cuda", dtype=torch.float64) if case["vectors"] else None
    return s


def run(state):
    c = state["case"]
    if c["op"] == "pairs":
        kl.kl_pairwise_noalloc(c["kernel"], 1.0, c["L"], state["tgt"], c["T"], state["src"], c["S"], state["X"],
                               c["S"], state["Y"], c["T"], c["k"], torch.cuda.current_stream())
        return state["Y"]
    h = state["handle"]
    N = h.N
    single = c["precision"] != "fp64"
    if c["op"] == "apply":
        call = kl.kl_apply_A if c["form"] == "A" else kl.kl_apply_Aprime
        call(h.h, state["X"], N, state["Y"], N, c["k"])
        return state["Y"].float() if single else state["Y"]
    if c["op"] == "zinv":
        kl.kl_apply_Zinv(h.h, state["X"], N, state["Y"], N, c["k"])
        return state["Y"]
    if c["op"] == "sample":
        out = state["out"]
        kl.kl_sample(h.h, c["M"], state["lam"], state["V"], N, state["xi"], c["M"], c["ns"], out, out.shape[1])
        return out
    tol = 1e-6 if single else 1e-12
    kl.kl_eigs(h.h, c["M"], tol, state["lam"], state["V"], N, 1)
    lam = state["lam"].astype(np.float32) if single else state["lam"].copy()
    return {"lam": lam, "V": state["V"]} if c["vectors"] else {"lam": lam}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

def _sizes(case):
    """(N, sources, targets)"""
    p = case["p"]
    N = S = T = 1
    exp = case["kernel"] in ("exp", "exp_sep")
    for d in (1, 2, 3):
        e = case[f"e{d}"]
        n, q = e + p, e * (p + 1)
        nt = e * p + 1 if exp else n
        if d == 1 and case["geometry"] == "half_annulus":
            n += p - 1
            nt += 1 if exp else p
        N, s = N * n, nt if case["method"] == "galerkin" else q
        S *= s
        T *= n if case["method"] == "collocation" else s
    return N, S, T


def work(case):
    k = case.get("k", 8)
    if case["op"] == "pairs":
        S, T = case["S"], case["T"]
        return {"bytes": 8 * (3 * (S + T) + k * (S + T)), "flops": S * T * (10 + 2 * k)}
    N, S, T = _sizes(case)
    p = case["p"]
    if case["op"] == "zinv":  # banded solves: two triangular sweeps per direction
        return {"bytes": 16 * N * k, "flops": N * k * 3 * 2 * (2 * p + 1)}
    if case["op"] == "sample":
        Q = case["e1"] * case["e2"] * case["e3"] * (p + 1) ** 3
        M, ns = case["M"], case["ns"]
        return {"bytes": 8 * (N * M + M * ns + Q * ns), "flops": 2 * N * M * ns + 2 * (p + 1) * Q * ns}
    # kernel values (once per symmetric pair) and the product with k columns
    values = S * (S + 1) / 2 if T == S else S * T
    one = values * 10 + S * T * 2 * k
    if case["op"] == "apply":
        return {"bytes": 8 * (2 * N * k + 3 * (S if S == T else S + T)), "flops": one}
    n = 4 + case["M"] // 8  # the fewest blocks a Krylov space of this size is built from
    return {"bytes": 8 * N * (case["M"] if case["vectors"] else 1), "flops": n * one}


# ---------------------------------------------------------------------------
# The same operators in 64 bits
# ---------------------------------------------------------------------------

def _knots(ne, p, cont, join=None):
    t = [0.0] * (p + 1)
    for i in range(1, ne):
        t += [i / ne] * (p - (join if join is not None and 2 * i == ne else cont))
    return np.array(t + [1.0] * (p + 1))


def _greville(t, p):
    n = len(t) - p - 1
    g = np.array([t[i + 1:i + p + 1].mean() for i in range(n)])
    # the point at the right end of its function's support (a C^-1 knot)
    left = np.array([t[i + 1] == t[i + p + 1] and t[i] < t[i + 1] and t[i + 1] < 1.0 for i in range(n)])
    return np.where(left, t[p:p + n], g) if left.any() else g, left


def _basis(t, p, x, left=None):
    x = np.asarray(x, dtype=np.float64)
    left = np.zeros(len(x), bool) if left is None else left
    cols = len(t) - 1
    last = max(i for i in range(cols) if t[i] < t[i + 1])
    B = np.zeros((len(x), cols))
    for i in range(cols):
        if t[i] < t[i + 1]:
            right = (t[i] <= x) & (x < t[i + 1]) | ((i == last) & (x == 1.0))
            B[:, i] = np.where(left, (t[i] < x) & (x <= t[i + 1]), right)
    for d in range(1, p + 1):
        C = np.zeros((len(x), cols - d))
        for i in range(cols - d):
            if t[i + d] > t[i]:
                C[:, i] += (x - t[i]) / (t[i + d] - t[i]) * B[:, i]
            if t[i + d + 1] > t[i + 1]:
                C[:, i] += (t[i + d + 1] - x) / (t[i + d + 1] - t[i + 1]) * B[:, i + 1]
        B = C
    return B


def _gauss(ne, n):
    x, w = np.polynomial.legendre.leggauss(n)
    lo = np.arange(ne)[:, None] / ne
    return (lo + (x + 1) / (2 * ne)).reshape(-1), np.tile(w / (2 * ne), ne)


def _arc(u):
    """Quarter arc: unit-circle point, d(angle)/du, weight function."""
    a, s = 1.0 - u, SQRT_HALF
    W = a * a + 2 * s * u * a + u * u
    nx, ny = a * a + 2 * s * u * a, 2 * s * u * a + u * u
    dx, dy, dW = -2 * a + 2 * s * (a - u), 2 * s * (a - u) + 2 * u, -2 * a + 2 * s * (a - u) + 2 * u
    cx, cy = nx / W, ny / W
    return cx, cy, cx * (dy - cy * dW) / W - cy * (dx - cx * dW) / W, W


def _angle(case, u):
    if case["geometry"] == "annulus":
        return _arc(u)
    second = u >= 0.5
    cx, cy, dt, W = _arc(np.where(second, 2 * u - 1, 2 * u))
    return np.where(second, -cy, cx), np.where(second, cx, cy), 2 * dt, W


def _map(case, u):
    """Points (n, 3) and det DF of the tensor grid of parameters u[0..2],
    direction 1 fastest."""
    g = _geo(case)
    U3, U2, U1 = (v.reshape(-1) for v in np.meshgrid(u[2], u[1], u[0], indexing="ij"))
    if case["geometry"] == "cube":
        return np.stack([U1, U2, U3], 1), np.ones(len(U1))
    if case["geometry"] == "projective_cube":
        D = 1.0 + g[0] * U1 + g[1] * U2 + g[2] * U3
        return np.stack([U1 / D, U2 / D, U3 / D], 1), 1.0 / D ** 4
    cx, cy, dt, _ = _angle(case, U1)
    r = g[0] + (g[1] - g[0]) * U2
    return np.stack([r * cx, r * cy, g[2] * U3], 1), r * dt * (g[1] - g[0]) * g[2]


def _weights(case, u):
    """NURBS weight function at the tensor grid."""
    U3, U2, U1 = (v.reshape(-1) for v in np.meshgrid(u[2], u[1], u[0], indexing="ij"))
    if case["geometry"] == "projective_cube":
        g = _geo(case)
        return 1.0 + g[0] * U1 + g[1] * U2 + g[2] * U3
    return np.ones(len(U1)) if case["geometry"] == "cube" else _angle(case, U1)[3]


def _cuda(a):
    t = torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64))
    return t.cuda() if torch.cuda.is_available() else t


def _kron(mats, X):
    """(M3 x M2 x M1) X for a block X of shape (k, n)."""
    n = [m.shape[1] for m in mats]
    Y = X.reshape(-1, n[2], n[1], n[0])
    Y = torch.einsum("ai,zkji->zkja", mats[0], Y)
    Y = torch.einsum("bj,zkja->zkba", mats[1], Y)
    return torch.einsum("ck,zkba->zcba", mats[2], Y).reshape(X.shape[0], -1)


def _gamma(kernel, L, P, Q):
    """Kernel matrix (rows P)."""
    d = [(P[:, j, None] - Q[None, :, j]) for j in range(3)]
    if kernel == "exp_sep":
        return torch.exp((d[0].abs_() + d[1].abs_() + d[2].abs_()).mul_(-1.0 / L))
    r2 = (d[0] * d[0]).add_(d[1] * d[1]).add_(d[2] * d[2])
    if kernel == "gauss":
        return r2.mul_(-1.0 / (L * L)).exp_()
    r = r2.sqrt_()
    if kernel == "exp":
        return r.mul_(-1.0 / L).exp_()
    r = r.mul_(math.sqrt(3.0) / L)
    return (1.0 + r).mul_(torch.exp(-r))


def _product(kernel, L, P, Q, X):
    """X (k, sources) -> (k, targets)"""
    step = max(1, int(2e8) // Q.shape[0])
    return torch.cat([X @ _gamma(kernel, L, P[i:i + step], Q).T for i in range(0, P.shape[0], step)], 1)


class Discrete:
    """1D factors, point sets and scalings of a case."""

    def __init__(self, case, L):
        p, self.case, self.L = case["p"], case, L
        half = case["geometry"] == "half_annulus"
        e = [case[f"e{d}"] for d in (1, 2, 3)]
        joins = [0 if half and d == 0 else None for d in range(3)]
        t = [_knots(e[d], p, p - 1, joins[d]) for d in range(3)]
        q, w = zip(*(_gauss(n, p + 1) for n in e))
        E = [_basis(t[d], p, q[d]) for d in range(3)]
        self.E = [_cuda(m) for m in E]
        W3 = np.einsum("k,j,i->kji", w[2], w[1], w[0]).reshape(-1)
        self.grid_points, det = _map(case, q)
        if case["method"] == "collocation":
            x = [_greville(t[d], p)[0] for d in range(3)]
            B = [_basis(t[d], p, x[d]) for d in range(3)]
            self.Binv = [_cuda(np.linalg.inv(b)) for b in B]
            self.Wc = _cuda(_weights(case, x))
            self.w = _kron(self.Binv, self.Wc[None])[0]
            self.Wq = _cuda(_weights(case, q))
            self.src, self.tgt = self.grid_points, _map(case, x)[0]
            self.F, self.scale = self.E, _cuda(W3 * det) / self.Wq
            return
        Z = [E[d].T @ (w[d][:, None] * E[d]) for d in range(3)]
        Lc = [np.linalg.cholesky(z) for z in Z]
        self.LinvT = [_cuda(np.linalg.inv(c).T) for c in Lc]
        self.Zinv = [_cuda(np.linalg.inv(z)) for z in Z]
        self.inv_sqrt_det = _cuda(det ** -0.5)
        if case["method"] == "galerkin_std":
            self.F, self.scale, self.src = self.E, _cuda(W3 * np.sqrt(det)), self.grid_points
        else:
            cont = 0 if case["kernel"] in ("exp", "exp_sep") else p - 1
            F, x = [], []
            for d in range(3):
                ti = _knots(e[d], p, cont, -1 if half and d == 0 else None)
                g, left = _greville(ti, p)
                Mx = _basis(ti, p, q[d]).T @ (w[d][:, None] * E[d])
                F.append(np.linalg.solve(_basis(ti, p, g, left).T, Mx))
                x.append(g)
            self.src, det = _map(case, x)
            self.F, self.scale = [_cuda(f) for f in F], _cuda(np.sqrt(det))
        self.tgt = self.src

    def zinv(self, X):
        if self.case["method"] == "collocation":
            return _kron(self.Binv, X * self.Wc) / self.w
        return _kron(self.Zinv, X)

    def apply(self, X, standard):
        col = self.case["method"] == "collocation"
        F = self.F
        if standard and not col:
            F = [f @ c for f, c in zip(F, self.LinvT)]
        U = _kron(F, X * self.w if col else X) * self.scale
        W = _product(self.case["kernel"], self.L, _cuda(self.tgt), _cuda(self.src), U)
        if col:
            return self.zinv(W) if standard else W
        return _kron([f.T for f in F], W * self.scale)

    def field(self, C):
        if self.case["method"] == "collocation":
            return _kron(self.E, C * self.w) / self.Wq
        return _kron(self.E, C) * self.inv_sqrt_det


def _exact_eigs(case, L):
    """Leading eigenvalues, and vectors where the case returns them."""
    M = case["M"]
    if case["geometry"] == "cube" and case["kernel"] in ("exp_sep", "gauss"):
        # a product kernel on the cube: the spectrum is that of the 1D factors
        one = []
        for d in (1, 2, 3):
            D = Discrete(dict(case, e1=case[f"e{d}"], e2=1, e3=1), L)
            x, y = (_cuda(np.pad(v[:len(np.unique(v[:, 0])), :1], ((0, 0), (0, 2)))) for v in (D.tgt, D.src))
            G = _gamma(case["kernel"], L, x, y)
            F = D.F[0]
            if case["method"] == "collocation":
                q = _cuda(_gauss(case[f"e{d}"], case["p"] + 1)[1])
                one.append(torch.linalg.eigvals(D.Binv[0] @ G @ (q[:, None] * F)).real)
            else:
                P = F @ D.LinvT[0]
                one.append(torch.linalg.eigvalsh(P.T @ G @ P))
        lam = torch.einsum("i,j,k->ijk", *one).reshape(-1).sort(descending=True).values[:M]
        return {"lam": lam.cpu().numpy(), **({"V": None} if case["vectors"] else {})}
    D = Discrete(case, L)
    n = _sizes(case)[0]
    if n > 2500:
        return None
    A = D.apply(torch.eye(n, dtype=torch.float64, device=D.E[0].device), True).T
    if case["method"] == "collocation":
        lam = torch.linalg.eigvals(A.cpu()).real.sort(descending=True).values[:M]
        return {"lam": lam.numpy(), **({"V": None} if case["vectors"] else {})}
    lam, Y = torch.linalg.eigh((A + A.T) / 2)
    out = {"lam": lam.flip(0)[:M].cpu().numpy()}
    if case["vectors"]:
        V = _kron(D.LinvT, Y.flip(1)[:, :M].T.contiguous())
        top = V.gather(1, V.abs().argmax(1, keepdim=True))
        out["V"] = V * top.sign()
    return out


def exact(case, seed):
    if case["op"] == "pairs":
        tgt, src = _points(case, seed)
        return _product(case["kernel"], case["L"], tgt.T, src.T, _normal(seed + 1, case["k"], case["S"]))
    if case["op"] == "eigs":
        return _exact_eigs(case, _length(case, seed))
    D = Discrete(case, case["L"])
    if case["op"] == "sample":
        lam, V, xi = _modes(case, seed)
        return D.field((xi * _cuda(np.sqrt(lam))) @ V)
    X = _normal(seed, case["k"], _sizes(case)[0])
    return D.zinv(X) if case["op"] == "zinv" else D.apply(X, case["form"] == "Aprime")
