"""Performance cases: what a program that uses this package has it do, through its public calls.

A case is one pass of one kind of work:
  op      Y = K X with the SG operator of one system (``sg_matvec``, ``sg_matvec_lowp``)
  pc      Z = P^-1 R with one system's preconditioner (``sg_precond_apply[_lowp]``)
  solve   ``sg_gmres_solve`` of all systems of a handle from a zero initial guess
  train   mini-batch Adam steps of the warm-start network (``learned.train``), then its weights

``listed()`` names the cases, ``draw()`` gives others of the same ranges, ``prepare()`` sets up the
handle (or the network) and the inputs of one pass from a seed, ``run()`` makes the pass,
``work()`` counts the bytes and operations that it cannot do without.  ``exact()`` gives the
result in 64 bits from plain torch and numpy: the problem (KL modes, chaos coefficients, Q1
stiffness stack, triple products), the ILU(0) preconditioners, the multigrid V-cycle, a conjugate
gradient solution and the network's training are written out below for that.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1910_11505_gb300 import learned, sg

DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------ the cases

def listed():
    c3 = dict(n=256, M=6, p=3, sigma=1.0, ell=0.5)
    c2 = dict(n=128, M=4, p=3, sigma=0.5, ell=0.5)
    return [
        # the operator on the smallest configuration: a launch and little else
        dict(name="op_n16_fp64", kind="op", n=16, M=2, p=2, sigma=0.5, ell=1.0, precision="fp64"),
        # FP64 operator of the 128 x 128 configuration: every step of an FP64 GMRES
        dict(name="op_n128_fp64", kind="op", precision="fp64", **c2),
        # FP32 operator of the largest configuration: the inner solver of the mixed form
        dict(name="op_n256_fp32", kind="op", precision="fp32", **c3),
        # odd mesh and the paper's own data (a_min 0.01, short correlation, coefficient degree 3)
        dict(name="op_n97_q3_fp32", kind="op", n=97, M=5, p=2, q=3, sigma=0.5, ell=0.1, a_min=0.01,
             precision="fp32"),
        # the default preconditioner (mean-based, natural-order ILU(0)) inside a mixed solve
        dict(name="pc_mean_n256_fp32", kind="pc", precond="mean", precision="fp32", **c3),
        # field-split Gauss-Seidel in FP64, natural order: the 128 x 128 configuration's own
        dict(name="pc_fsgs_n128_fp64", kind="pc", precond="fs_gs", precision="fp64", **c2),
        # the smoother of the paper's best method on the finest mesh (grouped field split)
        dict(name="pc_fg_n256_bf16", kind="pc", precond="fg", ilu_order="color4", precision="fp32",
             fg_bf16=1, **c3),
        # one V-cycle of G-M-F-I (field-split smoothing), for systems whose splits are too wide
        dict(name="pc_mg_fsgs_n128_fp32", kind="pc", precond="mg", mg_smoother="fs_gs",
             ilu_order="color4", coupling_bf16=1, precision="fp32", **c2),
        # a small FP64 solve with the defaults: latency of the whole GMRES loop
        dict(name="solve_n16_fp64", kind="solve", nsys=1, n=16, M=2, p=2, sigma=0.5, ell=1.0,
             precond="mean", precision="fp64", rtol=1e-10),
        # several mid-sized systems in one handle, G-M-Fg-I, mixed: training data of the warm start
        dict(name="solve_n64x4_mixed", kind="solve", nsys=4, n=64, M=4, p=3, sigma=0.8, ell=1.0,
             precond="mg", mg_smoother="fg", ilu_order="color4", precision="fp32", graphs=1,
             rtol=1e-10),
        # the largest configuration solved with G-M-Fg-I in the mixed form
        dict(name="solve_n256_mixed", kind="solve", nsys=1, precond="mg", mg_smoother="fg",
             ilu_order="color4", precision="fp32", fg_bf16=1, graphs=1, rtol=1e-10, **c3),
        # the warm-start network of the 64 x 64 systems: four epochs of mini-batches
        dict(name="train_n64_b256", kind="train", n=64, M=4, p=3, rows=2048, batch=256, steps=32,
             hidden=64),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    stoch = dict(sigma=round(rng.uniform(0.1, 1.0), 3), ell=round(rng.uniform(0.25, 2.0), 3))
    kind = rng.choice(["op", "op", "op", "pc", "pc", "pc", "solve", "solve", "train"])
    if kind == "train":
        batch = logint(16, 256)
        return dict(kind=kind, n=rng.choice([16, 32, 64]), M=rng.randint(2, 4), p=3,
                    rows=batch * (max(1, 128 // batch) + rng.randint(1, 6)), batch=batch,
                    steps=rng.randint(8, 32), hidden=rng.choice([32, 64]))
    if kind == "op":
        M, p = rng.choice([(2, 2), (3, 2), (4, 2), (5, 2), (6, 2), (2, 3), (3, 3), (4, 3), (5, 3),
                           (6, 3), (2, 4), (3, 4), (4, 4)])
        d = dict(kind=kind, n=logint(12, 256), M=M, p=p,
                 precision=rng.choice(["fp64", "fp32"]), **stoch)
        if rng.random() < 0.2:
            d["q"] = 3
        return d
    M, p = rng.choice([(2, 2), (3, 2), (4, 2), (5, 2), (6, 2), (2, 3), (3, 3), (4, 3)])
    if kind == "pc":
        pc = rng.choice(["mean", "fs_gs", "fg", "mg"])
        prec = rng.choice(["fp64", "fp32"])
        if pc in ("mean", "fs_gs"):
            return dict(kind=kind, precond=pc, n=logint(16, 160), M=M, p=p, precision=prec,
                        ilu_order=rng.choice(["natural", "color4"]), **stoch)
        if pc == "fg":
            return dict(kind=kind, precond=pc, n=logint(16, 160), M=M, p=p, precision=prec,
                        ilu_order="color4", fg_bf16=rng.randint(0, 1) if prec == "fp32" else 0,
                        **stoch)
        coarse = rng.choice([2, 3])
        return dict(kind=kind, precond=pc, n=coarse * 2 ** rng.randint(3, 6), mg_coarse=coarse,
                    mg_smoother=rng.choice(["fg", "fs_gs"]), M=M, p=p, precision=prec,
                    ilu_order="color4", **stoch)
    d = dict(kind=kind, nsys=rng.randint(1, 4), M=M, p=p, rtol=1e-10, **stoch)
    if rng.random() < 0.3:  # small systems with the default preconditioner
        return dict(d, n=rng.randint(10, 32), precond="mean", precision="fp64",
                    graphs=rng.randint(0, 1))
    return dict(d, n=2 ** rng.randint(4, 6 if d["nsys"] > 1 else 7), precond="mg",
                mg_smoother="fg", ilu_order="color4", precision=rng.choice(["fp64", "fp32"]),
                graphs=1)


# ------------------------------------------------------------------ one pass

SG_KEYS = ("n", "M", "p", "q", "a_min", "precond", "precision", "ilu_order", "fg_bf16",
           "coupling_bf16", "mg_smoother", "mg_coarse", "graphs", "rtol")


def _draws(case, seed):
    """(sigma, ell) of every system: the case's, each varied by up to 10 % from the seed."""
    r = np.random.default_rng([1910, seed])
    return [(case["sigma"] * r.uniform(0.9, 1.1), case["ell"] * r.uniform(0.9, 1.1))
            for _ in range(case.get("nsys", 1))]


def _field(case, seed):
    """Random chaos coefficients at every node, N x P in FP64, smaller for higher degrees (the
    fields and residuals that a solve meets)."""
    N, J = (case["n"] + 1) ** 2, _indices(case["M"], case["p"])
    gen = torch.Generator(device=DEV).manual_seed(seed)
    X = torch.randn(N, len(J), generator=gen, dtype=F64, device=DEV)
    return X * torch.tensor(0.5 ** J.sum(1), device=DEV)


def prepare(case, seed):
    if case["kind"] == "train":
        return _prepare_train(case, seed)
    prm = {k: case[k] for k in SG_KEYS if k in case}
    if case["kind"] == "op":
        prm["precond"] = "none"
    if case["kind"] == "solve":
        prm.update(restart=50, max_iters=400)
    h = sg.sg_setup([sg.sg_default_params(sigma=s, ell=l, **prm) for s, l in _draws(case, seed)])
    state = dict(kind=case["kind"], h=h, low=case["precision"] != "fp64")
    if case["kind"] == "solve":
        state["F"], state["X"] = [], []
        for i in range(h.nsys):
            N, P, _ = sg.sg_dims(h, i)
            F = torch.empty(N, P, dtype=F64, device=DEV)
            sg.sg_rhs(h, i, F)
            state["F"].append(F)
            state["X"].append(torch.zeros_like(F))
        return state
    X = _field(case, seed)
    state["X"] = X.float() if state["low"] else X
    state["Y"] = torch.empty_like(state["X"])
    return state


def run(state):
    kind = state["kind"]
    if kind == "op":
        (sg.sg_matvec_lowp if state["low"] else sg.sg_matvec)(state["h"], 0, state["X"], state["Y"])
        return state["Y"]
    if kind == "pc":
        apply = sg.sg_precond_apply_lowp if state["low"] else sg.sg_precond_apply
        apply(state["h"], 0, state["X"], state["Y"])
        return state["Y"]
    if kind == "solve":
        for x in state["X"]:
            x.zero_()
        sg.sg_gmres_solve(state["h"], state["F"], state["X"])
        return state["X"]
    learned.train(state["net"], state["Z"], state["T"], steps=state["steps"],
                  batch=state["batch"], lr=1e-3)
    return state["net"].get(0)


# ------------------------------------------------------------------ the warm-start network

IN = 6  # features at M = 4: sigma, ell and four KL weights; fewer modes leave the rest constant


def _net_data(case, seed):
    """Flat FP32 start parameters (NumPy), features Z and targets T (FP32, on the GPU): smooth
    combinations of 96 decaying modes, as solutions of nearby systems are."""
    D, hid = (case["n"] + 1) ** 2 * math.comb(case["M"] + case["p"], case["p"]), case["hidden"]
    r = np.random.default_rng([505, seed])
    parts = [r.uniform(-1, 1, (64, IN)) * math.sqrt(6.0 / (64 + IN)), np.zeros(64),
             r.uniform(-1, 1, (hid, 64)) * math.sqrt(6.0 / (hid + 64)), np.zeros(hid),
             np.zeros((D, hid)), np.zeros(D)]
    flat = np.concatenate([a.ravel() for a in parts]).astype(np.float32)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    Z = torch.rand(case["rows"], IN, generator=gen, device=DEV)
    mix = torch.randn(IN, 96, generator=gen, device=DEV)
    modes = torch.randn(96, D, generator=gen, device=DEV) * 0.01
    modes = modes / torch.arange(1, 97, device=DEV)[:, None]
    T = torch.sin(2 * Z @ mix + torch.arange(96, device=DEV)) @ modes
    return D, flat, Z, T.contiguous()


def _prepare_train(case, seed):
    D, flat, Z, T = _net_data(case, seed)
    net = sg.SGNet(IN, 64, case["hidden"], D, max_batch=case["batch"], bf16=True, seed=seed)
    net.set(0, flat)
    net.set_stats(Z, T)
    net.set_basis(T)
    return dict(kind="train", net=net, Z=Z, T=T, steps=case["steps"], batch=case["batch"])


def _exact_train(case, seed):
    D, flat, Z, T = _net_data(case, seed)
    hid = case["hidden"]
    Z = Z.to(F64)
    mu, sd = Z.mean(0), Z.std(0, unbiased=False).clamp_min(1e-6)
    b3 = T.to(F64).mean(0)
    basis = min(case["rows"], hid)
    Q, R = torch.linalg.qr((T[:basis].to(F64) - b3).T)
    Q = Q * torch.sign(torch.diagonal(R))
    scale = torch.stack([(Q.T @ (t.to(F64) - b3).T).abs().amax(1) for t in T.split(256)]).amax(0)
    W3 = torch.zeros(D, hid, dtype=F64, device=DEV)
    W3[:, :basis] = Q * (scale / 0.9)
    p0 = torch.tensor(flat[:64 * IN + 64 + hid * 64 + hid], dtype=F64, device=DEV)
    par = [a.reshape(s).clone().requires_grad_() for a, s in
           zip(p0.split([64 * IN, 64, hid * 64, hid]), [(64, IN), (64,), (hid, 64), (hid,)])]
    m, v = [torch.zeros_like(a) for a in par], [torch.zeros_like(a) for a in par]
    nb, order, rng = max(1, case["rows"] // case["batch"]), [], np.random.default_rng(7)
    for step in range(1, case["steps"] + 1):
        order = order or list(rng.permutation(nb))
        rows = slice((k := order.pop()) * case["batch"], (k + 1) * case["batch"])
        h = torch.tanh((Z[rows] - mu) / sd @ par[0].T + par[1])
        y = torch.tanh(h @ par[2].T + par[3]) @ W3.T + b3
        grads = torch.autograd.grad((y - T[rows].to(F64)).square().mean(), par)
        with torch.no_grad():
            for a, g, s, t in zip(par, grads, m, v):
                s.mul_(0.9).add_(0.1 * g)
                t.mul_(0.999).add_(0.001 * g * g)
                a -= 1e-3 * (s / (1 - 0.9 ** step)) / ((t / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return torch.cat([a.detach().ravel() for a in par] + [W3.ravel(), b3]).cpu().numpy()


# ------------------------------------------------------------------ what a pass cannot do without

def _triples(case):
    """(pairs, entries, L): the (k, b) pairs that meet a nonzero triple product, the nonzeros, and
    the coefficient's chaos terms."""
    G = _triple_products(_indices(case["M"], case.get("q") or 2 * case["p"]),
                         _indices(case["M"], case["p"]))
    return int((G != 0).any(1).sum()), int((G != 0).sum()), len(G)


def _op_work(case, n, s):
    """Operator: the stiffness stack (9 entries a node, L terms) read once, X read, Y written."""
    pairs, entries, L = _triples(case)
    N, P = (n + 1) ** 2, math.comb(case["M"] + case["p"], case["p"])
    return (3 * n + 1) ** 2 * L * s + 2 * N * P * s, 2 * N * (9 * pairs + entries)


def _pc_work(case, n, s, pc):
    """One level's block preconditioner: its factors read once, R read, Z written."""
    N, P = (n + 1) ** 2, math.comb(case["M"] + case["p"], case["p"])
    vec = 2 * N * P * s
    if pc == "mean":
        return 9 * N * s + vec, 2 * 9 * N * P
    if pc == "fg":
        fs = 2 if case.get("fg_bf16") else s
        return sum((b - a) ** 2 for a, b in _splits(case)) * 9 * N * fs + vec, \
            2 * 9 * N * sum((b - a) ** 2 for a, b in _splits(case))
    pairs, entries, L = _triples(case)  # fs_gs: every field's factors and the coupling's stack
    cs = 2 if case.get("coupling_bf16") else s
    return 9 * N * P * s + 9 * N * L * cs + vec, 2 * 9 * N * P + N * (9 * pairs + entries)


def work(case):
    s = 8 if case.get("precision", "fp64") == "fp64" else 4
    if case["kind"] == "train":
        D, B, hid = (case["n"] + 1) ** 2 * math.comb(case["M"] + case["p"], case["p"]), \
            case["batch"], case["hidden"]
        step = B * D * 4 + D * hid * 2 + D * 4
        return dict(bytes=case["steps"] * step + (D * (hid + 1) + 70 * hid) * 8,
                    flops=case["steps"] * 4 * B * D * hid)
    if case["kind"] == "op":
        b, f = _op_work(case, case["n"], s)
        return dict(bytes=b, flops=f)
    if case["precond"] == "mg":
        b = f = 0
        n = case["n"]
        while n > case.get("mg_coarse", 2):
            ob, of = _op_work(case, n, s)
            pb, pf = _pc_work(case, n, s, case["mg_smoother"])
            b, f, n = b + 2 * (ob + pb), f + 2 * (of + pf), n // 2
    else:
        b, f = _pc_work(case, case["n"], s, case["precond"])
    if case["kind"] == "pc":
        return dict(bytes=b, flops=f)
    # a solve: the iterations it needs in use (multigrid some nine; mean-based some forty), one
    # operator and one preconditioner each, and the FP64 residual of the solution
    ob, of = _op_work(case, case["n"], s)
    its = 9 if case["precond"] == "mg" else 40
    rb, rf = _op_work(case, case["n"], 8)
    return dict(bytes=case["nsys"] * (its * (b + ob) + rb), flops=case["nsys"] * (its * (f + of) + rf))


# ------------------------------------------------------------------ the problem in 64 bits

def _indices(M, p):
    """Multi-indices of total degree <= p in M variables, lexicographic, last index fastest."""
    out = [()]
    for _ in range(M):
        out = [a + (d,) for a in out for d in range(p - sum(a) + 1)]
    return np.array(out)


def _splits(case):
    """Field ranges of the grouped field split: groups of equal first index, a group that holds a
    multi-index of equal entries opens a split, another joins the one before."""
    J = _indices(case["M"], case["p"])
    out = []
    for d in range(case["p"] + 1):
        at = np.flatnonzero(J[:, 0] == d)
        if not out or (J[at] == J[at][:, :1]).all(1).any():
            out.append([at[0], at[-1] + 1])
        else:
            out[-1][1] = at[-1] + 1
    return [(int(a), int(b)) for a, b in out]


def _triple_products(Jq, Jp):
    """E[psi_q psi_a psi_b] of normalised Hermite polynomials, L x P x P."""
    f = math.factorial

    def one(i, j, k):
        s, odd = divmod(i + j + k, 2)
        if odd or s < max(i, j, k):
            return 0.0
        return math.sqrt(f(i) * f(j) * f(k)) / (f(s - i) * f(s - j) * f(s - k))

    dq, dp = Jq.max() + 1, Jp.max() + 1
    e = np.array([[[one(i, j, k) for k in range(dp)] for j in range(dp)] for i in range(dq)])
    G = np.ones((len(Jq), len(Jp), len(Jp)))
    for d in range(Jq.shape[1]):
        G *= e[Jq[:, d]][:, Jp[:, d]][:, :, Jp[:, d]]
    return G


def _kl_1d(ell, count):
    """1-D Karhunen-Loeve modes of exp(-|s-t|/ell) on [0, 1]: (w, odd, eigenvalue, norm)."""
    c, out = 1.0 / ell, []
    for k in range(count):
        odd = k % 2
        lo, hi = k * math.pi, (k + 1) * math.pi
        for _ in range(200):
            w = 0.5 * (lo + hi)
            v = w * math.cos(w / 2) + c * math.sin(w / 2) if odd else \
                c * math.cos(w / 2) - w * math.sin(w / 2)
            up = v > 0 if k % 4 < 2 else v < 0
            lo, hi = (w, hi) if up else (lo, w)
        out.append((w, odd, 2 * c / (w * w + c * c),
                    math.sqrt(0.5 + (-1) ** odd * math.sin(w) / (2 * w))))
    return out


def _blocks(case, n, sigma, ell):
    """K on an n x n mesh as one P x P block a node and 9-point neighbour: N x 9 x P x P."""
    M, m = case["M"], n + 1
    Jq = _indices(M, case.get("q") or 2 * case["p"])
    m1 = _kl_1d(ell, M + 1)
    top = sorted((-(a[2] * b[2]), i, j) for i, a in enumerate(m1) for j, b in enumerate(m1))[:M]
    r = math.sqrt(0.6)
    t, w = np.array([0.5 - 0.5 * r, 0.5, 0.5 + 0.5 * r]), np.array([5.0, 8.0, 5.0]) / 18.0
    x = ((np.arange(n)[:, None] + t) / n).ravel() - 0.5          # 3 n points of a line

    def line(mode):
        return (np.sin if mode[1] else np.cos)(mode[0] * x) / mode[3]

    # fields at the Gauss points, point (cell y, cell x, gy, gx)
    g = [math.sqrt(sigma * sigma * -v) * np.outer(line(m1[j]), line(m1[i])) for v, i, j in top]
    g = torch.tensor(np.array(g), device=DEV).reshape(M, n, 3, n, 3).permute(0, 1, 3, 2, 4)
    g = g.reshape(M, n * n, 9)
    a = torch.exp(0.5 * g.square().sum(0))[..., None].repeat(1, 1, len(Jq))
    for d in range(M):
        powers = torch.stack([g[d] ** k / math.sqrt(math.factorial(k))
                              for k in range(Jq.max() + 1)], -1)
        a *= powers[..., torch.tensor(Jq[:, d], device=DEV)]
    a[..., 0] += case.get("a_min", 0.0)
    A = torch.zeros(m, m, 9, len(Jq), dtype=F64, device=DEV)
    corner = [(0, 0), (1, 0), (0, 1), (1, 1)]                      # (x, y)
    for (ix, iy) in corner:
        for (jx, jy) in corner:
            c = np.empty(9)
            for q in range(9):
                xi, et = t[q % 3], t[q // 3]
                u, v = (xi if ix else 1 - xi), (et if iy else 1 - et)
                u2, v2 = (xi if jx else 1 - xi), (et if jy else 1 - et)
                c[q] = w[q % 3] * w[q // 3] * ((2 * ix - 1) * (2 * jx - 1) * v * v2
                                               + (2 * iy - 1) * (2 * jy - 1) * u * u2)
            val = torch.einsum("cgk,g->ck", a, torch.tensor(c, device=DEV)).reshape(n, n, -1)
            A[iy:iy + n, ix:ix + n, (jy - iy + 1) * 3 + jx - ix + 1] += val
    inner = torch.zeros(m + 2, m + 2, dtype=torch.bool, device=DEV)
    inner[2:-2, 2:-2] = True                                       # Dirichlet rows and columns
    for s in range(9):
        A[:, :, s] *= (inner[1:-1, 1:-1] & inner[s // 3:s // 3 + m, s % 3:s % 3 + m])[..., None]
    A[:, :, 4, 0] += (~inner[1:-1, 1:-1]).double()
    P = math.comb(M + case["p"], case["p"])
    G = torch.tensor(_triple_products(Jq, _indices(M, case["p"])), device=DEV)
    return (A.reshape(m * m * 9, -1) @ G.reshape(len(Jq), -1)).reshape(m * m, 9, P, P)


def _shifted(X, n, s):
    """X of the neighbour in slot s of every node (zero outside the mesh), N x P."""
    m = n + 1
    Xp = torch.nn.functional.pad(X.reshape(m, m, -1), (0, 0, 1, 1, 1, 1))
    return Xp[s // 3:s // 3 + m, s % 3:s % 3 + m].reshape(m * m, -1)


def _apply(K, X, n):
    return sum(torch.bmm(K[:, s], _shifted(X, n, s)[..., None])[..., 0] for s in range(9))


# ------------------------------------------------------------------ ILU(0) in 64 bits

class _ILU:
    """ILU(0) on the 9-point pattern in the natural or the four-colour node order, of blocks
    A: N x 9 x Q x Q (dense blocks) or N x 9 x F (F scalar matrices side by side)."""

    def __init__(self, A, n, order):
        m = n + 1
        self.A, self.dense = A.clone(), A.dim() == 4
        A = self.A
        self.D = torch.empty_like(A[:, 4])
        node = torch.arange(m * m, device=DEV)
        x, y = node % m, node // m
        self.nb = torch.stack([(x + s % 3 - 1).clamp(0, n) + m * (y + s // 3 - 1).clamp(0, n)
                               for s in range(9)], 1)
        key = x + 2 * y if order == "natural" else (x & 1) + 2 * (y & 1)
        self.levels = []
        for c in range(int(key.max()) + 1):
            if order == "natural":
                rank = list(range(9))
            else:  # colour of every slot's node, then its place
                rank = [(((c & 1) + s % 3 - 1) % 2 + 2 * (((c >> 1) + s // 3 - 1) % 2)) * 9 + s
                        for s in range(9)]
            mine = rank[4] if order == "natural" else c * 9
            low = sorted((s for s in range(9) if s != 4 and rank[s] < mine), key=lambda s: rank[s])
            high = [s for s in range(9) if s != 4 and s not in low]
            i = torch.nonzero(key == c)[:, 0]
            for s in low:
                k = self.nb[i, s]
                lik = self._mul(A[i, s], self.D[k])
                A[i, s] = lik
                for t in range(9):
                    dx, dy = t % 3 - s % 3, t // 3 - s // 3
                    if t != s and abs(dx) < 2 and abs(dy) < 2 and (t == 4 or rank[t] > rank[s]):
                        A[i, t] -= self._mul(lik, A[k, (dy + 1) * 3 + dx + 1])
            self.D[i] = torch.linalg.inv(A[i, 4]) if self.dense else 1.0 / A[i, 4]
            self.levels.append((i, low, high))

    def _mul(self, a, b):
        return torch.bmm(a, b) if self.dense else a * b

    def _vec(self, a, v):
        return torch.bmm(a, v[..., None])[..., 0] if self.dense else a * v

    def solve(self, R, col=slice(None)):
        """Z for the N x Q (or N x F) right-hand side; ``col``: the scalar matrices it is for."""
        part = (lambda a: a) if self.dense else (lambda a: a[:, col])
        Z = R.clone()
        for i, low, _ in self.levels:
            for s in low:
                Z[i] -= self._vec(part(self.A[i, s]), Z[self.nb[i, s]])
        for i, _, high in reversed(self.levels):
            v = Z[i]
            for s in high:
                v = v - self._vec(part(self.A[i, s]), Z[self.nb[i, s]])
            Z[i] = self._vec(part(self.D[i]), v)
        return Z


def _block_pc(case, K, n, pc):
    """R -> Z of one level's block preconditioner."""
    order = case.get("ilu_order", "natural")
    if pc == "mean":
        # E[psi_0 psi_0 psi_k] leaves only the mean stiffness in the first diagonal block
        f = _ILU(K[:, :, :1, 0], n, order)
        return lambda R: f.solve(R)
    if pc == "fs_gs":
        f = _ILU(torch.diagonal(K, dim1=2, dim2=3), n, order)

        def sweep(R):
            Z = torch.zeros_like(R)
            for a in range(R.shape[1]):
                r = R[:, a:a + 1].clone()
                if a:
                    for s in range(9):
                        r -= (K[:, s, a, :a] * _shifted(Z, n, s)[:, :a]).sum(1, keepdim=True)
                Z[:, a:a + 1] = f.solve(r, slice(a, a + 1))
            return Z
        return sweep
    ranges = _splits(case)
    fs = [_ILU(K[:, :, a:b, a:b], n, order) for a, b in ranges]

    def grouped(R):
        Z = torch.zeros_like(R)
        for (a, b), f in zip(ranges, fs):
            rhs = R - _apply(K, Z, n) if a else R
            Z[:, a:b] = f.solve(rhs[:, a:b].contiguous())
        return Z
    return grouped


def _vcycle(case, sigma, ell):
    sizes = [case["n"]]
    while sizes[-1] > case.get("mg_coarse", 2):
        sizes.append(sizes[-1] // 2)
    Ks = {n: _blocks(case, n, sigma, ell) for n in sizes}
    pcs = {n: _block_pc(case, Ks[n], n, case["mg_smoother"]) for n in sizes[:-1]}

    def up(u, n):  # bilinear interpolation from the interior of the n x n mesh to 2n x 2n
        m = n + 1
        c = torch.zeros(m, m, u.shape[1], dtype=F64, device=DEV)
        c[1:-1, 1:-1] = u.reshape(m, m, -1)[1:-1, 1:-1]
        f = torch.zeros(2 * n + 1, 2 * n + 1, u.shape[1], dtype=F64, device=DEV)
        f[::2, ::2] = c
        f[::2, 1::2] = 0.5 * (f[::2, :-1:2] + f[::2, 2::2])
        f[1::2] = 0.5 * (f[:-1:2] + f[2::2])
        return f.reshape(-1, u.shape[1])

    def down(r, n):  # its transpose
        m = n // 2 + 1
        f = r.reshape(n + 1, n + 1, -1)
        f = torch.nn.functional.pad(f, (0, 0, 1, 1, 1, 1))
        c = sum((1 - 0.5 * abs(dx)) * (1 - 0.5 * abs(dy)) * f[1 + dy:n + 2 + dy:2, 1 + dx:n + 2 + dx:2]
                for dx in (-1, 0, 1) for dy in (-1, 0, 1))
        out = torch.zeros(m, m, r.shape[1], dtype=F64, device=DEV)
        out[1:-1, 1:-1] = c[1:-1, 1:-1]
        return out.reshape(-1, r.shape[1])

    def cycle(b, n):
        K = Ks[n]
        if n == sizes[-1]:
            N, P = b.shape
            eye = torch.eye(N * P, dtype=F64, device=DEV).reshape(N * P, N, P)
            full = torch.stack([_apply(K, e, n).ravel() for e in eye], 1)
            m = torch.arange(N, device=DEV)
            inner = ((m % (n + 1) % n > 0) & (m // (n + 1) % n > 0)).repeat_interleave(P)
            u = torch.zeros(N * P, dtype=F64, device=DEV)
            u[inner] = torch.linalg.solve(full[inner][:, inner], b.ravel()[inner])
            return u.reshape(N, P)
        u = pcs[n](b)
        u = u + up(cycle(down(b - _apply(K, u, n), n), n // 2), n // 2)
        return u + pcs[n](b - _apply(K, u, n))

    return lambda R: cycle(R, case["n"])


# ------------------------------------------------------------------ solutions in 64 bits

def _solution(case, sigma, ell):
    """K u = F by conjugate gradients, preconditioned by the Laplacian's sine transform."""
    n, m = case["n"], case["n"] + 1
    K = _blocks(case, n, sigma, ell)
    P = K.shape[2]
    b = torch.zeros(m, m, P, dtype=F64, device=DEV)
    b[1:-1, 1:-1, 0] = 1.0 / (n * n)                    # the integral of a nodal basis function
    k = torch.arange(1, n, dtype=F64, device=DEV)
    S = torch.sin(math.pi / n * k[:, None] * k) * math.sqrt(2.0 / n)
    lam = 2 - 2 * torch.cos(math.pi / n * k)
    lam = (lam[:, None] + lam)[..., None]

    def pre(r):
        v = r.reshape(m, m, P)[1:-1, 1:-1]
        v = torch.einsum("ab,bcp,cd->adp", S, v, S) / lam
        out = torch.zeros_like(b)
        out[1:-1, 1:-1] = torch.einsum("ab,bcp,cd->adp", S, v, S)
        return out.reshape(-1, P)

    r = b.reshape(-1, P).clone()
    x, z = torch.zeros_like(r), pre(r)
    p, rz, stop = z, (r * z).sum(), 1e-15 * r.norm()
    for _ in range(500):
        q = _apply(K, p, n)
        alpha = rz / (p * q).sum()
        x, r = x + alpha * p, r - alpha * q
        if r.norm() < stop:
            break
        z = pre(r)
        rz, old = (r * z).sum(), rz
        p = z + rz / old * p
    return x


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    draws = _draws(case, seed)
    if case["kind"] == "solve":
        return [_solution(case, s, l) for s, l in draws]
    (s, l), X = draws[0], _field(case, seed)
    if case["precision"] != "fp64":
        X = X.float().to(F64)
    if case["kind"] == "op":
        return _apply(_blocks(case, case["n"], s, l), X, case["n"])
    if case["precond"] == "mg":
        return _vcycle(case, s, l)(X)
    if case["precond"] == "mean":  # one coefficient term and one field are enough for its factors
        K = _blocks(dict(case, p=0, q=0), case["n"], s, l)
    else:
        K = _blocks(case, case["n"], s, l)
    return _block_pc(case, K, case["n"], case["precond"])(X)
