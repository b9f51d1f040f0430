"""Cases of the measured work: what a program that solves differential matrix
equations with this library asks of it, through its public entry points.

Kinds:
  solve   ``Plan.solve`` of a dense plan (and the LQR gain of its result when
          the equation has a control): the plan is kept, each pass takes an
          initial state P0 through N composition steps
  plan    ``Plan(...)`` itself, with E_t and W_t exported: what a program pays
          once per problem and step length
  factor  ``LowRankPlan.solve`` (dense A) with the dense P as the output
  sparse  ``LowRankPlan.from_csr(...).solve`` on the stochastic heat problem
  serve   a batch of requests of mixed sizes through the server

Families of A: heat (5-point Dirichlet Laplacian), convdiff (with convection
(10, 10)), random (a stable dense matrix of any size).  The matrices' values
come from the seed, the sizes from the case.
"""
import math

import numpy as np
import torch

import paper_1805_08990_gb300 as dme

F64 = torch.float64
DEV = "cuda"


def listed():
    return [
        # a small control problem solved by itself: every launch and host call counts
        dict(name="dre_n81_fp64", kind="solve", family="convdiff", n=81, m=2, p=3, gen=False, prec="fp64",
             comp="strang", flows="F12 F3", T=0.0625, steps=16, fsal=False),
        # the plain Lyapunov configuration (heat equation on a 16 x 16 grid, h = T/100), each precision
        dict(name="dle_n256_fp64", kind="solve", family="heat", n=256, m=0, p=1, gen=False, prec="fp64",
             comp="strang", flows="F1 F2", T=0.1, steps=100, fsal=False),
        dict(name="dle_n256_split", kind="solve", family="heat", n=256, m=0, p=1, gen=False, prec="split_bf16",
             comp="strang", flows="F1 F2", T=0.1, steps=100, fsal=False),
        # the convection-diffusion Riccati configuration on a 32 x 32 grid, h = 1/256
        dict(name="dre_n1024_fp64", kind="solve", family="convdiff", n=1024, m=2, p=3, gen=False, prec="fp64",
             comp="strang", flows="F12 F3", T=8 / 256, steps=8, fsal=False),
        dict(name="dre_n1024_split", kind="solve", family="convdiff", n=1024, m=2, p=3, gen=False, prec="split_bf16",
             comp="strang", flows="F12 F3", T=64 / 256, steps=64, fsal=False),
        # the generalised Riccati equation on a 45 x 45 grid, an odd size (2025 unknowns), h = 1/128
        dict(name="gdre_n2025_fp64", kind="solve", family="convdiff", n=2025, m=4, p=5, gen=True, prec="fp64",
             comp="strang", flows="F12 F3 F4", T=2 / 128, steps=2, fsal=False),
        dict(name="gdre_n2025_split", kind="solve", family="convdiff", n=2025, m=4, p=5, gen=True, prec="split_bf16",
             comp="strang", flows="F12 F3 F4", T=16 / 128, steps=16, fsal=False),
        # the largest dense size in split precision: the heat Riccati problem on a 64 x 64 grid, h = 1/256
        dict(name="dre_n4096_split", kind="solve", family="heat", n=4096, m=8, p=8, gen=False, prec="split_bf16",
             comp="strang", flows="F12 F3", T=8 / 256, steps=8, fsal=False),
        # a plan: the exponential pair (E, W) of a step, which every new problem needs first
        dict(name="plan_n1024_fp64", kind="plan", family="convdiff", n=1024, m=2, p=3, gen=False, prec="fp64",
             comp="strang", flows="F12 F3", T=1.0, steps=256, fsal=False),
        # the factored path on a 48 x 48 grid, h = 1/256
        dict(name="factor_n2304_fp64", kind="factor", family="heat", n=2304, m=8, p=8, prec="fp64",
             comp="strang", flows="F1 F2 F3", T=8 / 256, steps=8),
        # the stochastic heat transfer problem with sparse A and S, h = 0.005
        dict(name="sparse_n3600", kind="sparse", n=3600, flows="F12 F3 F4", T=0.05, steps=10),
        # a queue of independent problems of mixed sizes, submitted together to a server
        dict(name="serve_12_split", kind="serve", count=12, n_min=32, n_max=768, prec="split_bf16", steps_min=50,
             steps_max=250, mix=3),
    ]


SCHEMES = {False: ["F12", "F1 F2"], True: ["F12 F3", "F1 F2 F3"]}
GEN = {False: ["F12 F4", "F1 F2 F4"], True: ["F12 F3 F4", "F12 F4 F3"]}


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def grid(n):
        return max(4, int(round(math.sqrt(n)))) ** 2

    kind = rng.choices(["solve", "plan", "factor", "sparse", "serve"], [7, 2, 1, 1, 1])[0]
    if kind == "solve":
        prec = rng.choice(["fp64", "fp64", "split_bf16"])
        n = size(24, 1600 if prec == "fp64" else 3000)
        family = rng.choice(["heat", "convdiff", "random"])
        if family != "random":
            n = grid(n)
        control, gen = rng.random() < 0.7, rng.random() < 0.25
        comp = rng.choice(["strang", "strang", "lie"])
        flows = rng.choice((GEN if gen else SCHEMES)[control])
        # steps: at most what the largest listed case computes
        limit = 4e10 if prec == "fp64" else 1.5e12
        steps = max(1, min(rng.choice([4, 16, 50, 100]), int(limit / (12.0 * n ** 3))))
        h = rng.choice([1 / 64, 1 / 256, 1 / 1024])
        fsal = comp == "strang" and " " in flows and rng.random() < 0.25
        return dict(kind=kind, family=family, n=n, m=rng.randint(1, 8) if control else 0, p=rng.randint(1, 8), gen=gen,
                    prec=prec, comp=comp, flows=flows, T=h * steps, steps=steps, fsal=fsal)
    if kind == "plan":
        family = rng.choice(["heat", "convdiff", "random"])
        n = size(32, 1100)
        if family != "random":
            n = grid(n)
        return dict(kind=kind, family=family, n=n, m=rng.randint(1, 8), p=rng.randint(1, 8), gen=False,
                    prec=rng.choice(["fp64", "split_bf16"]), comp="strang", flows="F12 F3", T=1.0,
                    steps=rng.choice([128, 256, 512]), fsal=False)
    if kind == "factor":
        return dict(kind=kind, family=rng.choice(["heat", "convdiff"]), n=grid(size(200, 2300)), m=rng.randint(1, 8),
                    p=rng.randint(1, 8), prec=rng.choice(["fp64", "split_bf16"]), comp="strang", flows="F1 F2 F3",
                    T=rng.choice([4, 6, 8]) / 256, steps=4)
    if kind == "sparse":
        steps = rng.choice([4, 6, 8, 10])
        return dict(kind=kind, n=grid(size(400, 3600)), flows=rng.choice(["F12 F3 F4", "F1 F2 F3 F4"]),
                    T=0.005 * steps, steps=steps)
    return dict(kind=kind, count=rng.randint(4, 12), n_min=32, n_max=rng.choice([200, 400, 600]),
                prec=rng.choice(["split_bf16", "fp64"]), steps_min=50, steps_max=rng.choice([80, 120]),
                mix=rng.randint(10, 10 ** 6))


# ------------------------------------------------------------------ inputs
def rng_of(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def uniform(g, *shape):
    return torch.rand(*shape, generator=g, dtype=F64, device=DEV)


def normal(g, *shape):
    return torch.randn(*shape, generator=g, dtype=F64, device=DEV)


def tridiag(nx, lo, mid, hi):
    one = torch.ones(nx - 1, dtype=F64, device=DEV)
    return torch.diag(one * lo, -1) + mid * torch.eye(nx, dtype=F64, device=DEV) + torch.diag(one * hi, 1)


def operator(family, n, g):
    """A (n x n): heat, convdiff (n a square) or random."""
    if family == "random":
        M = normal(g, n, n) / math.sqrt(n)
        return M - (M.abs().sum(0).max() + 1.0) * torch.eye(n, dtype=F64, device=DEV)
    nx = math.isqrt(n)
    assert nx * nx == n
    dx = 1.0 / (nx + 1)
    one = torch.eye(nx, dtype=F64, device=DEV)
    T1 = tridiag(nx, 1.0, -2.0, 1.0) / (dx * dx)
    if family == "convdiff":
        T1 = T1 - 10.0 * tridiag(nx, -1.0, 0.0, 1.0) / (2.0 * dx)
    return torch.kron(one, T1) + torch.kron(T1, one)


def problem(case, seed):
    """The data of a dense case: A, C, B, R, S and the initial state P0."""
    g = rng_of(seed)
    n, m = case["n"], case["m"]
    d = {"A": operator(case["family"], n, g)}
    d["S"] = 0.1 * normal(g, n, n) / math.sqrt(n) if case.get("gen") else None
    d["B"] = normal(g, n, m) if m else None
    d["R"] = torch.diag(0.5 + uniform(g, m)) if m else None
    d["C"] = uniform(g, case["p"], n)
    if case["kind"] == "solve":
        G = uniform(g, n, min(n, 64))
        P0 = G @ G.T / G.shape[1]
        d["P0"] = 0.5 * (P0 + P0.T)
    return d


class Csr:
    """A sparse matrix as its CSR arrays."""

    def __init__(self, n, rows, cols, vals):
        order = np.lexsort((cols, rows))
        self.shape = (n, n)
        self.indptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int32)
        self.indices = cols[order].astype(np.int32)
        self.data = vals[order].astype(np.float64)
        self.rows, self.cols, self.vals = rows, cols, vals

    def dense(self):
        M = torch.zeros(self.shape, dtype=F64, device=DEV)
        M[torch.as_tensor(self.rows, device=DEV), torch.as_tensor(self.cols, device=DEV)] = torch.as_tensor(self.vals, device=DEV)
        return M


def stochastic_heat(n, seed):
    """Heat transfer on an nx x nx grid, Dirichlet south and north, the control on the
    west edge, a Robin condition with noise on the east edge; the output C is a
    weighted mean whose smooth weights come from the seed."""
    nx = math.isqrt(n)
    dx = 1.0 / (nx + 1)
    i, j = np.arange(n) % nx, np.arange(n) // nx
    k = np.arange(n)
    diag = np.where(i == nx - 1, -3.0 + 0.25 * dx, -4.0)
    rows, cols, vals = [k], [k], [diag]
    for ok, off in ((i > 0, -1), (i < nx - 1, 1), (j > 0, -nx), (j < nx - 1, nx)):
        rows.append(k[ok])
        cols.append(k[ok] + off)
        vals.append(np.ones(ok.sum()))
    A = Csr(n, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals) / (dx * dx))
    east = k[i == nx - 1]
    S = Csr(n, east, east, np.full(nx, 0.5 / dx))
    B = np.zeros((n, 1))
    B[i == 0, 0] = 1.0 / (dx * dx)
    r = np.random.default_rng(seed)
    a, b, c = r.uniform(0.1, 0.9, 3)
    C = ((1.0 + c * np.cos(math.pi * ((i + 1) * dx * a + (j + 1) * dx * b))) / n)[None, :]
    return A, B, S, C


def requests(case, seed):
    """The requests of a serving case: sizes, horizons and step counts from the case's mix, values from the seed."""
    r = np.random.default_rng(case["mix"])
    out = []
    for k in range(case["count"]):
        n = int(round(math.exp(r.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        family = "heat" if r.integers(0, 2) else "random"
        if family == "heat":
            n = min(int(round(math.sqrt(n))), math.isqrt(case["n_max"])) ** 2
        out.append(dict(kind="request", family=family, n=n, m=int(r.integers(1, 9)), p=int(r.integers(1, 9)),
                        T=float(r.uniform(0.1, 10.0)), steps=int(r.integers(case["steps_min"], case["steps_max"] + 1)),
                        comp="strang", flows="F12 F3", seed=int(seed) * 1000 + k))
    return out


class Server:
    """A server handle that ends with its state."""

    def __init__(self):
        self.handle = dme.dme_server_create(16 << 30, 16)

    def __del__(self):
        try:
            dme.dme_server_destroy(self.handle)
        except Exception:
            pass


# ------------------------------------------------------------------ the calls
def build_plan(case, d):
    return dme.Plan(d["A"], C=d["C"], h=case["T"] / case["steps"], flows=case["flows"].split(), comp=case["comp"],
                    B=d["B"], R=d["R"], S=d["S"], prec=case["prec"], fsal=case["fsal"])


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "plan"):
        d = problem(case, seed)
        s = {"case": case, "d": d}
        if kind == "solve":
            s["plan"] = build_plan(case, d)
            s["P"] = torch.empty_like(d["P0"])
            if case["m"]:
                s["K"] = torch.empty(case["m"], case["n"], dtype=F64, device=DEV)
        else:
            s["E"] = torch.empty_like(d["A"])
            s["W"] = torch.empty_like(d["A"])
        return s
    if kind == "factor":
        d = problem(case, seed)
        plan = dme.LowRankPlan(d["A"], d["C"], h=case["T"] / case["steps"], flows=case["flows"].split(),
                               comp=case["comp"], B=d["B"], R=d["R"], prec=case["prec"])
        return {"case": case, "plan": plan, "P": torch.empty_like(d["A"])}
    if kind == "sparse":
        A, B, S, C = stochastic_heat(case["n"], seed)
        plan = dme.LowRankPlan.from_csr(A, C, h=case["T"] / case["steps"], flows=case["flows"].split(), comp="strang",
                                        B=B, R=np.eye(1), S_csr=S)
        return {"case": case, "plan": plan, "P": torch.empty(case["n"], case["n"], dtype=F64, device=DEV)}
    jobs = []
    for q in requests(case, seed):
        d = {k: None if v is None else v.cpu().numpy() for k, v in problem(q, q["seed"]).items()}
        desc = dme.make_desc(q["n"], m=q["m"], p=q["p"], eq=dme.DME_DRE, comp=q["comp"], flows=q["flows"].split(),
                             prec=case["prec"], h=q["T"] / q["steps"], q_is_factor=True)
        jobs.append((q, desc, d, np.zeros((q["n"], q["n"]))))
    return {"case": case, "server": Server(), "jobs": jobs}


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "solve":
        state["plan"].solve(state["d"]["P0"], case["T"], case["steps"], state["P"])
        if case["m"]:
            state["plan"].gain(state["P"], state["K"])
            return {"P": state["P"], "K": state["K"]}
        return {"P": state["P"]}
    if kind == "plan":
        with build_plan(case, state["d"]) as plan:
            plan.expm(0.5 * (case["T"] / case["steps"]), state["E"], state["W"])
        return {"E": state["E"], "W": state["W"]}
    if kind in ("factor", "sparse"):
        state["plan"].solve(case["T"], case["steps"], P_out=state["P"])
        return {"P": state["P"]}
    srv = state["server"].handle
    tickets = [dme.dme_submit(srv, desc, d["A"], d["C"], d["B"], d["R"], None, P0, q["T"], q["steps"])
               for q, desc, d, P0 in state["jobs"]]
    out = []
    for t, (q, desc, d, P0) in zip(tickets, state["jobs"]):
        P = np.empty((q["n"], q["n"]))
        dme.dme_poll(srv, t, P)
        out.append(P)
    return out


def sequence(comp, flows, h):
    """One step as (flow, length) pairs in the order they are applied."""
    if comp == "lie" or len(flows) == 1:
        return [(f, h) for f in flows]
    half = [(f, 0.5 * h) for f in flows[:-1]]
    return half + [(flows[-1], h)] + half[::-1]


def work(case):
    """Operations: n^3 multiply-adds for E^T (P E) in full and half of them for the symmetric
    product after it, the same per S P S^T, 2 n^2 m per product with B, the
    exponential's products and solves; bytes: each input and output once."""
    kind = case["kind"]
    if kind == "serve":
        r = [work(dict(q, kind="solve", gen=False)) for q in requests(case, 0)]
        return {"bytes": sum(x["bytes"] for x in r), "flops": sum(x["flops"] for x in r)}
    n = float(case["n"])
    flows = case["flows"].split()
    seq = sequence(case.get("comp", "strang"), flows, 1.0)
    if kind == "plan":  # 18 block products of the [13/13] approximant, two solves, a doubling per squaring (about 2)
        return {"flops": (18 * 2 + 2 * 8 / 3 + 2 * 5) * n ** 3, "bytes": 8.0 * (3 * n * n + 2 * n * case["m"] + n * case["p"])}
    if kind in ("factor", "sparse"):  # products with a factor of about 32 columns; P = L D L^T at the end
        r = 32.0
        per = 0.0
        for f, _ in seq:
            if f in ("F1", "F12"):
                per += 2.0 * n * n * r if kind == "factor" else 2.0 * 5 * n * r * 30
            elif f == "F3":
                per += 4.0 * n * r
            elif f == "F4":
                per += 4.0 * n * r
            per += 2.0 * n * r * r
        return {"flops": per * case["steps"] + n * n * r, "bytes": 8.0 * n * n * (2 if kind == "factor" else 1)}
    per = 0.0
    for f, _ in seq:
        if f in ("F1", "F12"):
            per += 3.0 * n ** 3
        elif f == "F4":
            per += 3.0 * n ** 3 * (2 if case["comp"] == "strang" else 1)
        elif f == "F3":
            per += 4.0 * n * n * case["m"]
        elif f == "F2":
            per += 2.0 * n * n
    return {"flops": per * case["steps"], "bytes": 8.0 * n * n * (5 if case.get("gen") else 4)}


# ------------------------------------------------------------------ the same in plain torch, 64 bits
def expm_action(At, X, t):
    """e^{t At} X by Taylor series over short substeps."""
    k = max(1, int(math.ceil(2.0 * t * float(At.abs().sum(1).max()))))
    for _ in range(k):
        term, X = X, X.clone()
        for j in range(1, 24):
            term = At @ term * (t / k / j)
            X += term
    return X


def ew(A, Q, t):
    """E = e^{tA} and W = int_0^t e^{sA^T} Q e^{sA} ds: Taylor series at a short length, then doublings."""
    s = max(0, int(math.ceil(math.log2(max(2.0 * t * float(A.abs().sum(0).max()), 1e-300)))))
    tau = math.ldexp(t, -s)
    n = A.shape[0]
    E = torch.eye(n, dtype=F64, device=DEV)
    term = E.clone()
    for j in range(1, 20):
        term = term @ A * (tau / j)
        E = E + term
    term = tau * Q
    W = term.clone()
    At = A.T.contiguous()
    for j in range(2, 26):
        V = At @ term
        term = (V + V.T) * (tau / j)
        W = W + term
    for _ in range(s):
        W = W + E.T @ (W @ E)
        W = 0.5 * (W + W.T)
        E = E @ E
    return E, W


def solve64(case, d, P, quadrature=False):
    """N steps of the scheme on dense matrices."""
    A, C = d["A"], d["C"]
    Q = C.T @ C
    Bt = None if d["B"] is None else d["B"] @ torch.linalg.inv(torch.linalg.cholesky(d["R"])).T
    seq = sequence(case.get("comp", "strang"), case["flows"].split(), case["T"] / case["steps"])
    pairs = {}
    for f, t in seq:
        if f in ("F1", "F12") and t not in pairs:
            E, W = ew(A, Q, t)
            if quadrature and f == "F12":  # the factored path's W: 7 Gauss-Legendre nodes
                x, w = np.polynomial.legendre.leggauss(7)
                W = torch.zeros_like(A)
                for xi, wi in zip(x, w):
                    L = expm_action(A.T.contiguous(), C.T.contiguous(), 0.5 * t * (1.0 + float(xi)))
                    W += (0.5 * t * float(wi)) * (L @ L.T)
            pairs[t] = E, W
    euler = case.get("comp", "strang") == "lie"
    for _ in range(case["steps"]):
        for f, t in seq:
            if f in ("F1", "F12"):
                E, W = pairs[t]
                P = E.T @ (P @ E)
                if f == "F12":
                    P = P + W
            elif f == "F2":
                P = P + t * Q
            elif f == "F3":
                Z = P @ Bt
                M = torch.eye(Bt.shape[1], dtype=F64, device=DEV) + t * (Bt.T @ Z)
                P = P - t * (Z @ torch.linalg.solve(M, Z.T))
            else:
                X = d["S"] @ P @ d["S"].T
                P = P + t * X if euler else P + t * X + (0.5 * t * t) * (d["S"] @ X @ d["S"].T)
            P = 0.5 * (P + P.T)
    return P


def gain64(d, P):
    return torch.linalg.solve(d["R"], d["B"].T @ P)


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = []
        for q in requests(case, seed):
            d = problem(q, q["seed"])
            out.append(solve64(q, d, torch.zeros_like(d["A"])).cpu().numpy())
        return out
    if kind == "sparse":
        A, B, S, C = stochastic_heat(case["n"], seed)
        t = lambda x: torch.as_tensor(x, dtype=F64, device=DEV)  # noqa: E731
        d = {"A": A.dense(), "B": t(B), "R": t(np.eye(1)), "S": S.dense(), "C": t(C)}
        return {"P": solve64(case, d, torch.zeros_like(d["A"]), quadrature=True)}
    d = problem(case, seed)
    if kind == "plan":
        E, W = ew(d["A"], d["C"].T @ d["C"], 0.5 * (case["T"] / case["steps"]))
        return {"E": E, "W": W}
    P = solve64(case, d, d["P0"] if kind == "solve" else torch.zeros_like(d["A"]), quadrature=True if kind == "factor" else False)
    return {"P": P, "K": gain64(d, P)} if kind == "solve" and case["m"] else {"P": P}
