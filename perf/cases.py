"""Performance cases: the work that a user of the pairing-Hamiltonian solver has it do.

Every case goes through the package's public entry points on inputs of the kinds
the workloads use (separable pairing strengths with noise, uniform single-particle
energies), from the smallest call to the largest one, in every arithmetic form.

  hx      one product y = H x on the device (``pairdiag_hx_dev``): the step that an
          iterative solver, a propagator or a response calculation repeats
  trunc   the same product in the truncated model space (Dimension_Limit)
  solve   a whole ground state (``pairdiag_ground_state_dev``)
  batch   ground states of many uneven problems from host arrays, as a mean-field
          loop asks for them (``pairdiag_batch_ground_state``)
  mlp     one forward and backward pass of the warm-start network from host rows
          (``pairdiag_mlp_loss_grad``), the training direction
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2001_01978_gb300 as pd

PRECISION = {"fp64": pd.PD_PREC_FP64, "fp32": pd.PD_PREC_MIXED, "ff": pd.PD_HX_FLOATFLOAT}
X_TYPE = {"fp64": torch.float64, "fp32": torch.float32, "ff": torch.float32}
Y_TYPE = {"fp64": torch.float64, "fp32": torch.float32, "ff": torch.float64}
MAX_NNZ = {"fp64": 4.0e9, "fp32": 3.5e10, "ff": 8.0e9}      # drawn products stay below the largest listed one


# ------------------------------------------------------------------ cases ---
def listed():
    return [
        # the smallest call: a light nucleus' shell, doubly degenerate orbits (dim 924); launch and host latency
        {"name": "hx_fp64_o12_n6", "kind": "hx", "prec": "fp64", "omega": 12, "n": 6},
        # a small odd size of a mean-field loop (dim 12376), off half filling
        {"name": "hx_fp32_o17_n6", "kind": "hx", "prec": "fp32", "omega": 17, "n": 6},
        # the default benchmark's product (dim 2.7e6), in the mixed form's FP32 vectors
        {"name": "hx_fp32_o24_n12", "kind": "hx", "prec": "fp32", "omega": 24, "n": 12},
        # the same product in plain FP64, the form that every other is judged by
        {"name": "hx_fp64_o24_n12", "kind": "hx", "prec": "fp64", "omega": 24, "n": 12},
        # the FP64-accurate product of an FP32 vector (the mixed form's refinement), off half filling (dim 497420)
        {"name": "hx_ff_o22_n9", "kind": "hx", "prec": "ff", "omega": 22, "n": 9},
        # the largest product: dim 1.55e8, the size of the paper's timed large run
        {"name": "hx_fp32_o30_n15", "kind": "hx", "prec": "fp32", "omega": 30, "n": 15},
        # low filling, as in the paper's Table 3 (dim 5.2e7): many short basis blocks
        {"name": "hx_fp32_o34_n9", "kind": "hx", "prec": "fp32", "omega": 34, "n": 9},
        # the truncated model space: about a tenth of the states of Omega = 24 kept
        {"name": "trunc_fp32_o24_n12", "kind": "trunc", "prec": "fp32", "omega": 24, "n": 12, "limit": 250_000},
        # energy of the default benchmark's size in the mixed form, tightly converged
        {"name": "solve_mixed_o24_n12", "kind": "solve", "prec": "fp32", "omega": 24, "n": 12, "tol": 1e-6},
        # eigenpair of a mid-size problem (dim 43758) in plain FP64 to the last digits
        {"name": "solve_fp64_o18_n8", "kind": "solve", "prec": "fp64", "omega": 18, "n": 8, "tol": 1e-12},
        # one call of a mean-field loop: 96 uneven problems, Omega 10..22, host arrays in and energies out
        {"name": "batch_mixed_96", "kind": "batch", "prec": "fp32", "count": 96, "lo": 10, "hi": 22, "tol": 1e-6},
        # gradient of the warm-start network on its training set's size (3333 orbit rows)
        {"name": "mlp_grad_3333", "kind": "mlp", "rows": 3333},
    ]


def _draw_size(rng, lo_dim, hi_dim, omega_lo, omega_hi, max_nnz):
    """(omega, n) with a dimension near a log-uniform target."""
    target = math.exp(rng.uniform(math.log(lo_dim), math.log(hi_dim)))
    every = [(o, n) for o in range(omega_lo, omega_hi + 1) for n in range(2, o - 1)
             if math.comb(o, n) * n * (o - n) <= max_nnz]
    near = [(o, n) for o, n in every if target / 1.6 <= math.comb(o, n) <= target * 1.6]
    if not near:
        near = [min(every, key=lambda s: abs(math.log(math.comb(*s) / target)))]
    return near[rng.randrange(len(near))]


def draw(rng):
    kind = rng.choices(["hx", "trunc", "solve", "batch", "mlp"], [10, 2, 4, 2, 1])[0]
    if kind == "hx":
        prec = rng.choices(["fp32", "fp64", "ff"], [5, 3, 2])[0]
        omega, n = _draw_size(rng, 300, 1.3e8, 10, 34, MAX_NNZ[prec])
        return {"kind": "hx", "prec": prec, "omega": omega, "n": n}
    if kind == "trunc":
        prec = rng.choice(["fp32", "fp64"])
        omega, n = _draw_size(rng, 5e4, 5e6, 18, 28, 1.0e9)
        return {"kind": "trunc", "prec": prec, "omega": omega, "n": n,
                "limit": int(math.comb(omega, n) * rng.uniform(0.03, 0.6))}
    if kind == "solve":
        if rng.random() < 0.5:
            omega, n = _draw_size(rng, 1000, 2.0e6, 11, 24, 4.0e8)
            return {"kind": "solve", "prec": "fp32", "omega": omega, "n": n, "tol": 1e-6}
        omega, n = _draw_size(rng, 500, 2.0e5, 11, 22, 4.0e7)
        return {"kind": "solve", "prec": "fp64", "omega": omega, "n": n, "tol": 1e-12}
    if kind == "batch":
        lo = rng.randint(9, 13)
        return {"kind": "batch", "prec": rng.choice(["fp32", "fp64"]), "count": int(round(math.exp(rng.uniform(math.log(6), math.log(96))))),
                "lo": lo, "hi": lo + rng.randint(3, 7), "tol": 1e-6}
    return {"kind": "mlp", "rows": int(round(math.exp(rng.uniform(math.log(10), math.log(6000)))))}


# ----------------------------------------------------------------- inputs ---
def _noise(rng, omega, sigma=0.05):
    eta = np.triu(rng.normal(0.0, sigma, size=(omega, omega)))
    return eta + np.triu(eta, 1).T


def _hamiltonian(omega, rng, sort=True):
    """e ~ U[-10,10], G_ij = -g_i g_j + eta_ij with g ~ U[0.3,0.7] and symmetric eta ~ N(0, 0.05^2)."""
    e = rng.uniform(-10.0, 10.0, size=omega)
    if sort:
        e = np.sort(e)
    g = rng.uniform(0.3, 0.7, size=omega)
    return e, -np.outer(g, g) + _noise(rng, omega)


def _batch_problems(case, seed):
    rng = np.random.default_rng([seed, 3])
    probs = []
    for _ in range(case["count"]):
        omega = int(rng.integers(case["lo"], case["hi"] + 1))
        n = min(max(omega // 2 + int(rng.integers(-3, 4)), 1), omega - 1)
        e, G = _hamiltonian(omega, rng, sort=False)
        probs.append((omega, n, e, G))
    return probs


def _mlp_rows(case, seed):
    rng = np.random.default_rng([seed, 4])
    rows, X = case["rows"], []
    have = 0
    while have < rows:                       # feature rows of problems of the training sizes
        omega = int(rng.integers(10, 19))
        n = min(max(omega // 2 + int(rng.integers(-3, 4)), 1), omega - 1)
        e, G = _hamiltonian(omega, rng, sort=False)
        X.append(pd.pairdiag_mlp_features(omega, n, e, G))
        have += omega
    X = np.ascontiguousarray(np.concatenate(X)[:rows])
    t = (-1.5 * X[:, 0] + rng.normal(0.0, 0.1, size=rows)).astype(np.float32)
    theta = (rng.normal(0.0, 0.12, size=pd.pairdiag_mlp_num_params())).astype(np.float32)
    return X, t, theta


def _vector(dim, dtype, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed * 7 + 11)
    x = torch.randn(dim, dtype=dtype, device="cuda", generator=gen)
    return x * (1.0 / math.sqrt(dim))


class _State:
    """What the program keeps: the solver or network handle, its inputs, its output buffers."""

    def __init__(self, case):
        self.case, self.solver, self.net = case, None, None

    def __del__(self):
        try:
            if self.solver is not None:
                self.solver.close()
            if self.net is not None:
                pd.pairdiag_mlp_destroy(self.net)
        except Exception:
            pass


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "batch":
        s.problems = _batch_problems(case, seed)
        s.opt = pd.pairdiag_default_options(precision=PRECISION[case["prec"]], seed=seed % 1000 + 1)
        return s
    if kind == "mlp":
        s.X, s.t, theta = _mlp_rows(case, seed)
        s.net = pd.pairdiag_mlp_create(1)
        pd.pairdiag_mlp_set_params(s.net, theta)
        return s
    omega, n, prec = case["omega"], case["n"], case["prec"]
    e, G = _hamiltonian(omega, np.random.default_rng([seed, 1]))
    form = pd.PD_PREC_FP64 if prec == "fp64" else pd.PD_PREC_MIXED
    s.solver = pd.Solver(omega, n, e, G, precision=form, seed=seed % 1000 + 1)
    h = s.solver.h
    pd.pairdiag_set_stream(h, torch.cuda.current_stream())
    if kind == "solve":
        s.vec = torch.empty(s.solver.dim, dtype=torch.float64, device="cuda") if prec == "fp64" else None
        return s
    if kind == "trunc":
        pd.pairdiag_truncate(h, case["limit"])
    s.x = _vector(s.solver.dim, X_TYPE[prec], seed)
    s.y = torch.empty(s.solver.dim, dtype=Y_TYPE[prec], device="cuda")
    return s


# --------------------------------------------------------------- one pass ---
def run(s):
    case = s.case
    kind = case["kind"]
    if kind in ("hx", "trunc"):
        pd.pairdiag_hx_dev(s.solver.h, PRECISION[case["prec"]], s.x, s.y)
        return s.y
    if kind == "solve":
        r = pd.pairdiag_ground_state_dev(s.solver.h, case["tol"], s.vec)
        return {"e0": r["e0"]} if s.vec is None else {"e0": r["e0"], "vec": s.vec}
    if kind == "batch":
        r = pd.pairdiag_batch_ground_state(s.problems, case["tol"], s.opt)
        return {"e0": r["e0"]}
    loss, grad = pd.pairdiag_mlp_loss_grad(s.net, s.X, s.t)
    return {"loss": loss, "grad": grad}


# ------------------------------------------------------------------- work ---
def work(case):
    kind = case["kind"]
    if kind == "mlp":
        r = case["rows"]
        macs = r * (16 * 128 + 2 * 128 * 128 + 128)          # forward; the backward pass takes twice that
        params = 16 * 128 + 2 * 128 * 128 + 128 * 4 + 1
        return {"bytes": float(4 * (17 * r + params)), "flops": float(2 * macs * 3)}
    if kind == "batch":
        steps = 60                                           # about what such problems need
        dims = [(math.comb(o, o // 2), (o // 2) * (o - o // 2)) for o in range(case["lo"], case["hi"] + 1)]
        dim = case["count"] * sum(d for d, _ in dims) / len(dims)
        nnz = case["count"] * sum(d * k for d, k in dims) / len(dims)
        es = 8 if case["prec"] == "fp64" else 4
        return {"bytes": steps * dim * es * 4.0, "flops": steps * 2.0 * nnz}
    omega, n, prec = case["omega"], case["n"], case["prec"]
    dim = math.comb(omega, n)
    nnz = dim * n * (omega - n)
    es = 8 if prec == "fp64" else 4
    if kind == "solve":                                      # a product and the newest three vectors per Lanczos step
        steps = 80
        return {"bytes": steps * dim * es * 4.0, "flops": steps * 2.0 * nnz}
    if kind == "trunc":                                      # the kept part of the rows and of each row
        share = min(1.0, case["limit"] / dim)
        return {"bytes": dim * share * es * 2.0, "flops": 2.0 * nnz * share * share}
    return {"bytes": float(dim * (es + (8 if prec == "ff" else es))), "flops": 2.0 * nnz}


# ------------------------------------------------------ 64-bit references ---
def _binom(omega):
    return torch.tensor([[math.comb(p, j) if j <= p else 0 for p in range(omega + 1)] for j in range(omega + 2)],
                        dtype=torch.int64, device="cuda")


def _states(omega, n):
    """Every omega-bit word with n set bits, ascending (colexicographic unranking of 0..dim-1)."""
    r = torch.arange(math.comb(omega, n), dtype=torch.int64, device="cuda")
    w = torch.zeros_like(r)
    B = _binom(omega)
    for j in range(n, 0, -1):
        p = torch.searchsorted(B[j], r, right=True) - 1
        r = r - B[j][p]
        w |= torch.ones_like(p) << p
    return w


class _Rank:
    """Index of a word among the ascending n-bit words, from tables of its two halves."""

    def __init__(self, omega, n):
        self.cut = omega // 2
        lo, hi = 1 << self.cut, 1 << (omega - self.cut)
        self.mask = lo - 1
        low, high = np.zeros(lo, dtype=np.int64), np.zeros(hi, dtype=np.int64)
        count = np.array([bin(i).count("1") for i in range(max(lo, hi))])
        for p in range(self.cut):
            at = np.nonzero(np.arange(lo) >> p & 1)[0]
            order = count[at & ((1 << p) - 1)] + 1
            low[at] += np.array([math.comb(p, int(j)) for j in range(self.cut + 2)])[order]
        for p in range(omega - self.cut):
            at = np.nonzero(np.arange(hi) >> p & 1)[0]
            order = n - count[at] + count[at & ((1 << p) - 1)] + 1
            table = np.array([math.comb(self.cut + p, j) for j in range(n + 2)])
            high[at] += np.where((order >= 0) & (order <= n), table[np.clip(order, 0, n + 1)], 0)
        self.low, self.high = torch.from_numpy(low).cuda(), torch.from_numpy(high).cuda()

    def __call__(self, w):
        return self.high[w >> self.cut] + self.low[w & self.mask]


def _diagonal(omega, e, G, w):
    d = torch.zeros(w.numel(), dtype=torch.float64, device="cuda")
    for p in range(omega):
        d += (w >> p & 1).double() * float(2.0 * e[p] + G[p, p])
    return d


def _product(omega, n, e, G, x, kept=None):
    """H x in 64 bits; kept: the indices of a truncated space's states (x and the result hold those)."""
    w = _states(omega, n)
    rank = _Rank(omega, n)
    full = x
    if kept is not None:
        full = torch.zeros(w.numel(), dtype=torch.float64, device="cuda")
        full[kept] = x
        w = w[kept]
    y = _diagonal(omega, e, G, w) * x
    for i in range(omega):
        for j in range(i):
            at = torch.nonzero(((w >> i) ^ (w >> j)) & 1).squeeze(1)
            if at.numel():
                y.index_add_(0, at, full[rank(w[at] ^ ((1 << i) | (1 << j)))] * float(G[i, j]))
    return y


def _kept(omega, n, e, G, limit, bins=100_000_000):
    d = _diagonal(omega, e, G, _states(omega, n))
    lo, hi = d.min(), d.max()
    b = torch.clamp(torch.floor((d - lo) / (hi - lo) * float(bins)), max=bins - 1)
    cut = torch.sort(b).values[min(limit, d.numel()) - 1]
    return torch.nonzero(b <= cut).squeeze(1)


def _lowest(omega, n, e, G):
    """Lowest eigenvalue: Lanczos with full reorthogonalisation on the explicit rows, 64 bits."""
    w = _states(omega, n)
    rank = _Rank(omega, n)
    dim, hops = w.numel(), n * (omega - n)
    diag = _diagonal(omega, e, G, w)
    idx = torch.zeros((dim, max(hops, 1)), dtype=torch.int64, device="cuda")
    val = torch.zeros((dim, max(hops, 1)), dtype=torch.float64, device="cuda")
    fill = torch.zeros(dim, dtype=torch.int64, device="cuda")
    for i in range(omega):
        for j in range(i):
            at = torch.nonzero(((w >> i) ^ (w >> j)) & 1).squeeze(1)
            idx[at, fill[at]] = rank(w[at] ^ ((1 << i) | (1 << j)))
            val[at, fill[at]] = float(G[i, j])
            fill[at] += 1
    m = min(dim, 160)
    Q = torch.zeros((m, dim), dtype=torch.float64, device="cuda")
    q = torch.exp(-(diag - diag.min()) / 4.0) + 1e-3
    Q[0] = q / q.norm()
    alpha, beta = [], []
    for k in range(m):
        p = diag * Q[k] + (val * Q[k][idx]).sum(1)
        alpha.append(float(p @ Q[k]))
        for _ in range(2):
            p -= Q[:k + 1].T @ (Q[:k + 1] @ p)
        b = float(p.norm())
        if k % 10 == 9 or k == m - 1 or b < 1e-12 * abs(alpha[0]):
            T = np.diag(alpha) + np.diag(beta, 1) + np.diag(beta, -1)
            th, s = np.linalg.eigh(T)
            if k == m - 1 or b * abs(s[-1, 0]) < 1e-11 * abs(th[0]):
                return float(th[0])
        beta.append(b)
        Q[k + 1] = p / b
    return float(th[0])


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return {"e0": np.array([_lowest(o, n, e, G) for o, n, e, G in _batch_problems(case, seed)])}
    if kind == "mlp":
        return _mlp_exact(*_mlp_rows(case, seed))
    omega, n = case["omega"], case["n"]
    e, G = _hamiltonian(omega, np.random.default_rng([seed, 1]))
    if kind == "solve":
        e0 = _lowest(omega, n, e, G)
        return {"e0": e0} if case["prec"] != "fp64" else {"e0": e0, "vec": None}     # the vector's sign is free
    kept = _kept(omega, n, e, G, case["limit"]) if kind == "trunc" else None
    dim = math.comb(omega, n) if kept is None else kept.numel()
    x = _vector(dim, X_TYPE[case["prec"]], seed).double()
    return _product(omega, n, e, G, x, kept)


def _mlp_exact(X, t, theta):
    X, t = torch.from_numpy(X).double().cuda(), torch.from_numpy(t).double().cuda()
    p = torch.from_numpy(theta).double().cuda().requires_grad_(True)
    at, parts = 0, []
    for rows, cols in ((16, 128), (1, 128), (128, 128), (1, 128), (128, 128), (1, 128), (128, 1), (1, 1)):
        parts.append(p[at:at + rows * cols].reshape(rows, cols))
        at += rows * cols
    a = X
    for W, b in zip(parts[0:6:2], parts[1:6:2]):
        a = torch.nn.functional.silu(a @ W + b)
    loss = ((a @ parts[6] + parts[7]).squeeze(1) - t).square().mean()
    loss.backward()
    return {"loss": float(loss.detach()), "grad": p.grad}
