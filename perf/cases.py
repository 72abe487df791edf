"""What this framework is timed on: its public entry points over the sizes, precisions and
options that a DG-CheFSI calculation uses (the workloads of paper_1606_03416_gb300/inputs.py,
their reduced copies, and odd and uneven sizes between them).

Every input comes from its seed; blocks of states are drawn on the GPU, Hamiltonians by the
repository's generator. A "warm" block is what a cycle meets after the first ones: plain
FP32 torch iterations of the same method (filter, QR, Rayleigh-Ritz) from a random block."""
import math

import numpy as np
import torch

from paper_1606_03416_gb300 import dgchefsi as D
from paper_1606_03416_gb300 import inputs as G
from paper_1606_03416_gb300.autograd import band_energy

DEV = "cuda"
SCALES = {"27": {1: 0.05, 2: 0.02, 3: 0.01}, "9": {1: 0.05, 2: 0.02}}
KT = 0.01
A0, B = -1.7, 44.0  # the generator's spectrum: diagonal blocks in [-1, 40] plus the couplings


def listed():
    return [
        # The Lanczos bound of one cycle on the tiny 2x2x2 workload: all latency.
        {"name": "bounds_tiny_2x2x2", "kind": "bounds", "gx": 2, "gy": 2, "gz": 2, "lo": 32, "hi": 32, "k": 10},
        # The tiny workload's filter (48 states, degree 10): launches and latency of one filter call.
        {"name": "filter_tiny_2x2x2", "kind": "filter", "prec": "bf16x3", "graph": False, "gx": 2, "gy": 2, "gz": 2,
         "lo": 32, "hi": 32, "Ns": 48, "m": 10},
        # The default precision on the reduced bulk copy: a user who asks for nothing.
        {"name": "filter_f64_bulk3d_4x4x4", "kind": "filter", "prec": "f64", "graph": False, "gx": 4, "gy": 4, "gz": 4,
         "lo": 64, "hi": 64, "Ns": 300, "m": 12},
        # The headline: one filter call of the 8x8x8 bulk workload in split BF16.
        {"name": "filter_bulk3d_8x8x8", "kind": "filter", "prec": "bf16x3", "graph": False, "gx": 8, "gy": 8, "gz": 8,
         "lo": 64, "hi": 64, "Ns": 4096, "m": 20},
        # The 2D sheet with uneven elements, replayed from its graph in TF32: the largest block.
        {"name": "filter_sheet2d_24x20_tf32", "kind": "filter", "prec": "tf32", "graph": True, "gx": 24, "gy": 20,
         "gz": 1, "lo": 40, "hi": 120, "Ns": 21554, "m": 16},
        # One whole warm cycle of the 8x8x8 workload with the subspace problem on the tensor cores.
        {"name": "cycle_bulk3d_8x8x8", "kind": "cycle", "prec": "bf16x3", "products": "sliced_bf16", "gx": 8, "gy": 8,
         "gz": 8, "lo": 64, "hi": 64, "Ns": 4096, "m": 20, "warm": 4},
        # Rayleigh-Ritz alone as it is by default (FP64 products), a small uneven sheet, an odd block.
        {"name": "rayleigh_ritz_sheet2d_8x6", "kind": "rr", "products": "f64", "gx": 8, "gy": 6, "gz": 1, "lo": 40,
         "hi": 120, "Ns": 401, "m": 16, "warm": 2},
        # The eigensolve of a converging cycle's projected H (nearly diagonal, a coupled top block).
        {"name": "eigh_2500", "kind": "eigh", "n": 2500, "top": 120},
        # The Cholesky factor's inverse of Cholesky-QR, an order that is no power of two.
        {"name": "cholesky_inverse_2999", "kind": "chol", "n": 2999},
        # One FP64 product from slices, ragged in every size, K past one 4096-long chunk.
        {"name": "sliced_gemm_1537x2001x9000", "kind": "gemm", "rows": 1537, "cols": 2001, "K": 9000, "b_rows": True},
        # Band energy forward and backward (the differentiated cycle) in its default precision, a reduced bulk copy.
        {"name": "band_energy_grad_4x4x4", "kind": "grad", "prec": "f64", "products": "sliced_bf16", "gx": 4,
         "gy": 4, "gz": 4, "lo": 40, "hi": 40, "Ns": 300, "m": 8, "warm": 2},
        # Re-alignment to the next SCF step's basis, once per SCF step (216 grid points per element).
        {"name": "realign_6x6x6", "kind": "realign", "gx": 6, "gy": 6, "gz": 6, "lo": 40, "hi": 72, "Ns": 1001,
         "points": 216},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, largest):
    if rng.random() < 0.35:
        g = (rng.randint(3, 2 * largest), rng.randint(3, 2 * largest), 1)
    else:
        g = tuple(rng.randint(2, largest) for _ in range(3))
    lo = rng.choice([16, 32, 40, 48, 64])
    return {"gx": g[0], "gy": g[1], "gz": g[2], "lo": lo, "hi": lo if rng.random() < 0.6 else min(120, 2 * lo + 7)}


def _least_N(c):
    return c["gx"] * c["gy"] * c["gz"] * c["lo"]


def draw(rng):
    kind = rng.choice(["bounds", "filter", "filter", "cycle", "rr", "eigh", "chol", "gemm", "grad", "realign"])
    if kind == "bounds":
        return {"kind": kind, **_grid(rng, 8), "k": rng.randint(4, 20)}
    if kind == "filter":
        prec = rng.choice(["bf16x3", "bf16x3", "tf32", "bf16", "f64"])
        c = {"kind": kind, "prec": prec, "graph": rng.random() < 0.3, **_grid(rng, 4 if prec == "f64" else 7)}
        return {**c, "Ns": min(_log(rng, 16, 400 if prec == "f64" else 3000), _least_N(c)), "m": rng.randint(6, 24)}
    if kind in ("cycle", "rr"):
        c = {"kind": kind, "products": rng.choice(["sliced_bf16", "sliced_bf16", "f64"]), **_grid(rng, 5)}
        if kind == "cycle":
            c["prec"] = rng.choice(["bf16x3", "bf16x3", "f64"])
        # about the lowest states of every element, as in the workloads (Ns / N is 0.1 to 0.25 there)
        return {**c, "Ns": max(16, int(min(900, _least_N(c) * rng.uniform(0.08, 0.22)))), "m": rng.randint(10, 20),
                "warm": 3}
    if kind == "eigh":
        n = _log(rng, 300, 3000)
        return {"kind": kind, "n": n, "top": rng.randint(0, n // 10)}
    if kind == "chol":
        return {"kind": kind, "n": _log(rng, 100, 3500)}
    if kind == "gemm":
        return {"kind": kind, "rows": _log(rng, 200, 4000), "cols": _log(rng, 200, 4000), "K": _log(rng, 100, 20000),
                "b_rows": rng.random() < 0.6}
    if kind == "grad":
        c = {"kind": kind, "prec": "f64", "products": rng.choice(["sliced_bf16", "f64"]), **_grid(rng, 4)}
        return {**c, "Ns": max(16, int(min(300, _least_N(c) * rng.uniform(0.08, 0.2)))), "m": rng.randint(5, 10), "warm": 2}
    return {"kind": kind, **_grid(rng, 6), "Ns": _log(rng, 40, 1500), "points": rng.randint(125, 343)}


# ---------------------------------------------------------------- inputs


def _config(c, seed):
    stencil = "9" if c["gz"] == 1 else "27"
    return G.ProblemConfig(name="case", grid=(c["gx"], c["gy"], c["gz"]), periodic=(True, True, c["gz"] > 1),
                           stencil=stencil, nb=c["lo"] if c["lo"] == c["hi"] else (c["lo"], c["hi"]), Ns=1, m=1, Ne=1.0,
                           kT=KT, scales=SCALES[stencil], seed=seed)


def _hamiltonian(c, seed):
    """The repository's generator. Where the element sizes are drawn they are the case's, not the
    seed's: there the seed flips the signs of basis functions (H -> D H D, D = diag(+-1))."""
    if c["lo"] == c["hi"]:
        return G.make_blocks(_config(c, seed))
    H = G.make_blocks(_config(c, 0))
    sign = np.random.default_rng(seed + 31).choice([-1.0, 1.0], size=H.N)
    off = np.concatenate([[0], np.cumsum(H.nb)])
    for K in range(H.M):
        for e in range(int(H.row_ptr[K]), int(H.row_ptr[K + 1])):
            L, n, q = int(H.col[e]), int(H.nb[K]), int(H.nb[H.col[e]])
            blk = H.values[int(H.blk_off[e]):int(H.blk_off[e]) + n * q].reshape(n, q)
            blk *= sign[off[K]:off[K + 1], None] * sign[None, off[L]:off[L + 1]]
    return H


def _gauss(shape, seed, dtype=torch.float64):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return torch.randn(shape, generator=g, device=DEV, dtype=dtype)


class _TorchH:
    """H as rows of blocks in plain torch: (H X^T)^T for state-major X, element by element."""

    def __init__(self, H, dtype):
        off = np.concatenate([[0], np.cumsum(H.nb)])
        vals = torch.from_numpy(H.values).to(DEV).to(dtype)
        self.rows, self.N = [], H.N
        for K in range(H.M):
            e0, e1, n = int(H.row_ptr[K]), int(H.row_ptr[K + 1]), int(H.nb[K])
            cols = np.concatenate([np.arange(off[j], off[j + 1]) for j in H.col[e0:e1]])
            w = [int(H.nb[j]) for j in H.col[e0:e1]]
            blk = torch.cat([vals[int(H.blk_off[e]):int(H.blk_off[e]) + n * q].view(n, q) for e, q in zip(range(e0, e1), w)], 1)
            self.rows.append((int(off[K]), int(off[K + 1]), torch.from_numpy(cols).to(DEV), blk.T.contiguous()))

    def apply(self, X):
        Y = torch.empty_like(X)
        for lo, hi, cols, blk in self.rows:
            Y[:, lo:hi] = X[:, cols] @ blk
        return Y

    def filter(self, X, m, a, b, a0):
        e, c = 0.5 * (b - a), 0.5 * (b + a)
        s1 = e / (a0 - c)
        prev, cur, s = X, (self.apply(X) - c * X) * (s1 / e), s1
        for _ in range(1, m):
            sn = 1.0 / (2.0 / s1 - s)
            prev, cur, s = cur, (self.apply(cur) - c * cur) * (2.0 * sn / e) - (s * sn) * prev, sn
        return cur

    def bound(self, v, k):
        """(upper bound, smallest Ritz value) of k Lanczos steps with full re-orthogonalisation."""
        V = [v / v.norm()]
        al, be = [], []
        for j in range(min(k, self.N)):
            w = self.apply(V[j][None])[0]
            if j:
                w = w - be[-1] * V[j - 1]
            al.append(float(torch.dot(V[j], w)))
            w = w - al[-1] * V[j]
            Q = torch.stack(V)
            w = w - Q.T @ (Q @ w)
            be.append(float(w.norm()))
            if be[-1] == 0.0:
                break
            V.append(w / be[-1])
        t = np.linalg.eigvalsh(np.diag(al) + np.diag(be[:len(al) - 1], 1) + np.diag(be[:len(al) - 1], -1))
        return float(t[-1] + abs(be[len(al) - 1])), float(t[0])


def _warm(H, Ns, m, seed, cycles):
    """(X, Ritz values) after `cycles` FP32 cycles from a random block: orthonormal to FP32, float64 outside."""
    T = _TorchH(H, torch.float32)
    X = _gauss((Ns, H.N), seed, torch.float32)
    a0, a = A0, A0 + (B - A0) * Ns / H.N
    for _ in range(cycles):
        Q = torch.linalg.qr(T.filter(X, m, a, B, a0).T)[0].T.contiguous()
        S = Q @ T.apply(Q).T
        w, V = torch.linalg.eigh(0.5 * (S + S.T))
        X = V.T @ Q
        a0, a = float(w[0]), float(w[-1])
    return X.double().contiguous(), w.double().cpu().numpy()


def _electrons(Ns):
    return G.default_ne(Ns) if Ns > 40 else float(Ns)


def _near_diagonal(c, seed):
    d = G.clustered_spectrum(c["n"], seed=seed)
    return G.near_diagonal_symmetric(d, 2e-8, c["top"], 1e-4, seed=seed)


def _gram_like(c, seed):
    """The overlap matrix of filtered states: rows of very different norms, well conditioned beside that."""
    n = c["n"]
    A = _gauss((n, n + 64), seed)
    S = A @ A.T / (n + 64) + 0.5 * torch.eye(n, dtype=torch.float64, device=DEV)
    d = torch.exp(torch.linspace(5.0, -5.0, n, dtype=torch.float64, device=DEV))
    return S * d[:, None] * d[None, :]


def _gemm_operands(c, seed):
    """States with amplitudes over three orders, as a filtered block has."""
    amp = lambda n, s: torch.exp(2.0 * _gauss((n, 1), s))  # noqa: E731
    A = _gauss((c["rows"], c["K"]), seed) * amp(c["rows"], seed + 101)
    Bm = _gauss((c["cols"], c["K"]) if c["b_rows"] else (c["K"], c["cols"]), seed + 202)
    return A, Bm * amp(Bm.shape[0], seed + 303)


def _realign_sizes(c):
    rng = np.random.default_rng(17)
    M = c["gx"] * c["gy"] * c["gz"]
    nb_old = rng.integers(c["lo"], c["hi"] + 1, size=M).astype(np.int32)
    nr = np.full(M, max(c["points"], c["hi"]), dtype=np.int32)
    return nb_old, nr


def _bases(nb, nr, seed):
    """Packed R_K x J_K sample blocks with columns of unit norm on average."""
    n = int((nr.astype(np.int64) * nb).sum())
    return _gauss((n,), seed) / math.sqrt(float(nr[0]))


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    if kind in ("eigh", "chol", "gemm"):  # a context of the tiny workload carries the settings and workspace
        s["ctx"] = D.Context(G.make_blocks(G.CONFIGS["tiny_2x2x2"]))
        s["ctx"].set_subspace_products("sliced_bf16", 10)
        if kind == "eigh":
            s["A"] = torch.from_numpy(_near_diagonal(c, seed)).to(DEV)
        elif kind == "chol":
            s["S"] = _gram_like(c, seed)
        else:
            s["A"], s["B"] = _gemm_operands(c, seed)
        return s
    H = _hamiltonian(c, seed)
    s["ctx"] = ctx = D.Context(H)
    if kind == "bounds":
        s["v"] = _gauss((H.N,), seed + 1)
    elif kind == "filter":
        s["X"] = _gauss((c["Ns"], H.N), seed + 1)
        s["Y"] = torch.empty_like(s["X"])
        s["a"] = A0 + (B - A0) * max(c["Ns"] / H.N, 0.02)
    elif kind == "realign":
        s["nb_old"], s["nr"] = _realign_sizes(c)
        s["V_old"], s["V_new"] = _bases(s["nb_old"], s["nr"], seed + 2), _bases(np.asarray(H.nb), s["nr"], seed + 3)
        s["X"] = _gauss((c["Ns"], int(s["nb_old"].sum())), seed + 1)
    else:
        ctx.set_subspace_products(c["products"], 10)
        s["X"], s["ritz"] = _warm(H, c["Ns"], c["m"], seed + 1, c["warm"])
        s["Ne"] = _electrons(c["Ns"])
        if kind == "cycle":
            s["v"] = _gauss((H.N,), seed + 2)
        elif kind == "grad":
            s["values"] = torch.from_numpy(H.values).to(DEV).requires_grad_(True)
            s["X"].requires_grad_(True)
    return s


def _aligned(X, before):
    """Each state with the sign it had in the block before (an eigenvector's sign is free; states are followed by it)."""
    return X.mul_(torch.where(torch.linalg.vecdot(X, before) < 0, -1.0, 1.0)[:, None])


def run(s):
    c, ctx = s["case"], s["ctx"]
    kind = c["kind"]
    if kind == "bounds":
        return np.array(ctx.bounds(s["v"], c["k"]))
    if kind == "filter":
        f = ctx.filter_graph if c["graph"] else ctx.filter
        return f(s["X"], c["m"], s["a"], B, A0, prec=c["prec"], Y=s["Y"])
    if kind == "eigh":
        w, V = ctx.subspace_eigh(s["A"].clone())  # in place in the library
        return {"w": w, "V": V}
    if kind == "chol":
        return torch.tril(ctx.cholesky_inverse(s["S"].clone()))
    if kind == "gemm":
        return ctx.sliced_gemm(s["A"], s["B"], b_rows=c["b_rows"])
    if kind == "realign":
        return ctx.realign(s["X"], s["nb_old"], s["nr"], s["V_old"], s["V_new"])
    if kind == "rr":
        Y = s["X"].clone()  # becomes X_new
        ritz = ctx.rayleigh_ritz(Y)
        f, mu = ctx.occupations(ritz, s["Ne"], KT)
        return {"X": _aligned(Y, s["X"]), "ritz": ritz, "f": f, "mu": mu, "P": ctx.density_blocks(Y, f)}
    if kind == "cycle":
        X = s["X"].clone()  # becomes X_new
        out = ctx.cycle(X, c["m"], s["Ne"], KT, v0=s["v"], prev_ritz=s["ritz"], prec=c["prec"])
        return {"X": _aligned(X, s["X"]), "ritz": out["ritz"], "f": out["f"], "mu": out["mu"], "P": out["P"]}
    E = band_energy(s["values"], s["X"], ctx, c["m"], float(s["ritz"][-1]), B, float(s["ritz"][0]), s["Ne"], KT,
                    prec=c["prec"])
    gv, gx = torch.autograd.grad(E, (s["values"], s["X"]))
    return {"E": E.detach(), "H_bar": gv, "X_bar": gx}


# ---------------------------------------------------------------- what a pass cannot do without


def _sizes(c):
    """(N, stored entries of H, sum of n_K^2) at the mean element size."""
    n = 0.5 * (c["lo"] + c["hi"])
    M = c["gx"] * c["gy"] * c["gz"]
    reach = lambda g: min(g, 3)  # noqa: E731
    nbrs = reach(c["gx"]) * reach(c["gy"]) * reach(c["gz"])
    return M * n, M * nbrs * n * n, M * n * n


def work(case):
    c, kind = case, case["kind"]
    if kind == "eigh":
        return {"bytes": 16.0 * c["n"] ** 2, "flops": 9.0 * c["n"] ** 3}
    if kind == "chol":
        return {"bytes": 8.0 * c["n"] ** 2, "flops": 2.0 / 3.0 * c["n"] ** 3}
    if kind == "gemm":
        r, q, k = c["rows"], c["cols"], c["K"]
        return {"bytes": 8.0 * (r * k + q * k + r * q), "flops": 2.0 * r * q * k}
    N, nnz, dens = _sizes(c)
    if kind == "bounds":
        return {"bytes": 8.0 * nnz, "flops": 2.0 * nnz * c["k"]}
    Ns = c["Ns"]
    if kind == "filter":
        return {"bytes": 8.0 * (nnz + 2 * Ns * N), "flops": 2.0 * nnz * Ns * c["m"]}
    if kind == "realign":
        return {"bytes": 8.0 * (2 * Ns * N + 2 * c["points"] * N), "flops": 2.0 * dens * (Ns + c["points"])}
    # Gram, Y U^-1 and projected H by their triangles, the rotation, Cholesky and eigensolve
    rr = 5.0 * Ns * Ns * N + (2.0 / 3.0 + 9.0) * Ns ** 3 + 2.0 * nnz * Ns
    if kind == "rr":
        return {"bytes": 8.0 * (nnz + 2 * Ns * N + dens), "flops": rr + 2.0 * dens * Ns}
    if kind == "cycle":
        return {"bytes": 8.0 * (nnz + 2 * Ns * N + dens), "flops": rr + 2.0 * dens * Ns + 2.0 * nnz * Ns * c["m"]}
    # forward, forward again with its iterates kept, and the reverse recurrence with its outer products
    return {"bytes": 8.0 * (2 * nnz + 2 * Ns * N), "flops": 2 * rr + 2.0 * nnz * Ns * c["m"] * 4}


# ---------------------------------------------------------------- the same in 64 bits


def _occupations(ritz, Ne):
    w = ritz.cpu().numpy()
    f = lambda mu: 1.0 / (1.0 + np.exp(np.clip((w - mu) / KT, -700, 700)))  # noqa: E731
    lo, hi = w.min() - 50 * KT, w.max() + 50 * KT
    for _ in range(200):
        mu = 0.5 * (lo + hi)
        lo, hi = (mu, hi) if 2 * f(mu).sum() < Ne else (lo, mu)
    return torch.from_numpy(f(mu)).to(DEV), torch.tensor([mu], dtype=torch.float64, device=DEV)


def _rayleigh_ritz(T, H, Y, Ne):
    L = torch.linalg.cholesky(Y @ Y.T)
    Q = torch.linalg.solve_triangular(L, Y, upper=False)
    S = Q @ T.apply(Q).T
    w, V = torch.linalg.eigh(0.5 * (S + S.T))
    X = V.T @ Q
    f, mu = _occupations(w, Ne)
    off = np.concatenate([[0], np.cumsum(H.nb)])
    P = torch.cat([(X[:, a:b].T @ (f[:, None] * X[:, a:b])).reshape(-1) for a, b in zip(off[:-1], off[1:])])
    # the states' signs are free: only what does not depend on them is given
    return {"X": None, "ritz": w, "f": f, "mu": mu, "P": P}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "eigh":
        A = torch.from_numpy(_near_diagonal(c, seed)).to(DEV)
        return {"w": torch.linalg.eigvalsh(A), "V": None}
    if kind == "chol":
        S = _gram_like(c, seed)
        L = torch.linalg.cholesky(S)
        return torch.linalg.solve_triangular(L, torch.eye(c["n"], dtype=torch.float64, device=DEV), upper=False)
    if kind == "gemm":
        A, Bm = _gemm_operands(c, seed)
        return A @ (Bm.T if c["b_rows"] else Bm)
    H = _hamiltonian(c, seed)
    if kind == "realign":
        nb_old, nr = _realign_sizes(c)
        Vo, Vn = _bases(nb_old, nr, seed + 2), _bases(np.asarray(H.nb), nr, seed + 3)
        X = _gauss((c["Ns"], int(nb_old.sum())), seed + 1)
        out, x, o, n = [], 0, 0, 0
        for K in range(H.M):
            R, j0, j1 = int(nr[K]), int(nb_old[K]), int(H.nb[K])
            Tk = Vn[n:n + R * j1].view(R, j1).T @ Vo[o:o + R * j0].view(R, j0)
            out.append(X[:, x:x + j0] @ Tk.T)
            x, o, n = x + j0, o + R * j0, n + R * j1
        return torch.cat(out, 1)
    N, nnz, _ = _sizes(c)
    if kind == "grad" or (kind == "filter" and 2.0 * nnz * c["Ns"] * c["m"] > 1.2e13):
        return None
    T = _TorchH(H, torch.float64)
    if kind == "bounds":
        return np.array(T.bound(_gauss((H.N,), seed + 1), c["k"]))
    if kind == "filter":
        return T.filter(_gauss((c["Ns"], H.N), seed + 1), c["m"], A0 + (B - A0) * max(c["Ns"] / H.N, 0.02), B, A0)
    X, ritz = _warm(H, c["Ns"], c["m"], seed + 1, c["warm"])
    if kind == "cycle":
        b = T.bound(_gauss((H.N,), seed + 2), 10)[0]
        X = T.filter(X, c["m"], float(ritz[-1]), b, float(ritz[0]))
    return _rayleigh_ritz(T, H, X, _electrons(c["Ns"]))
