"""Kernels at the edges of their tiles and of the ranges their dispatch takes them for,
against the CPU oracle or a closed form, within the bounds of each path (FP64_TOL,
SPLIT_TOL)."""
import numpy as np
import pytest
import scipy.fft
import scipy.linalg
import scipy.sparse as sp
import torch

import dme_workloads as W
import oracle as O
import paper_1805_08990_gb300 as dme
from gpu_util import FP64_TOL, SPLIT_TOL, dev, host, rel, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _gpu():
    require_gpu()


def _stable(n, seed):
    r = np.random.default_rng(seed)
    return r.standard_normal((n, n)) / np.sqrt(n) - 2.5 * np.eye(n)


# 8 x 8 tiles of the FP64 products (n < 192), full and triangular, and the flows around them
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 17, 31, 33, 64, 65, 100, 127, 129, 191])
def test_small_fp64_steps_match_oracle(n):
    r = np.random.default_rng(n)
    A, C, S = _stable(n, n), r.standard_normal((2, n)), 0.1 * r.standard_normal((n, n)) / np.sqrt(n)
    P0 = W.random_psd(n, 3)
    plan = dme.Plan(dev(A), C=dev(C), h=0.05, flows=["F12", "F4"], S=dev(S))
    ref = O.Plan(A, C.T @ C, None, None, S)
    for flow in ("F1", "F12", "F4"):
        P = dev(P0)
        plan.apply(flow, 0.05, P)
        assert rel(host(P), ref.apply(flow, 0.05, P0, "midpoint")) < FP64_TOL
        assert torch.equal(P, P.T)


# T3: every m of the register kernels and the first of the general one, n at the edges of the
# row blocks, of the 32-wide update tiles and beyond one row block per part
@pytest.mark.parametrize("n", [1, 3, 33, 255, 257, 1025, 2431, 2433])
@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 7, 8, 9, 16, 32])
def test_riccati_flow_matches_oracle(n, m):
    r = np.random.default_rng(100 * n + m)
    B, R = r.standard_normal((n, m)), np.diag(0.5 + r.uniform(size=m))
    G = r.standard_normal((n, 8))
    P0 = G @ G.T / n
    plan = dme.Plan(dev(np.diag(-1.0 - r.uniform(size=n))), C=dev(np.ones((1, n))), h=0.1, flows=["F3"], comp="lie",
                    B=dev(B), R=dev(R))
    P = dev(P0)
    plan.apply("F3", 0.1, P)
    Z = P0 @ B                                   # (I + t P B R^-1 B^T)^{-1} P by Woodbury
    ref = P0 - 0.1 * Z @ np.linalg.solve(R + 0.1 * B.T @ Z, Z.T)
    assert rel(host(P), ref) < FP64_TOL
    assert torch.equal(P, P.T)


# T3 of split plans: FP64 kernels or tensor products, by n and m
@pytest.mark.parametrize("n,m", [(1536, 5), (1537, 3), (1537, 4), (1537, 5), (1601, 9), (3600, 4), (3601, 4)])
def test_riccati_flow_of_split_plans_matches_formula(n, m):
    g = torch.Generator(device="cuda")
    g.manual_seed(n + m)
    B = torch.randn(n, m, generator=g, dtype=torch.float64, device="cuda")
    R = torch.diag(0.5 + torch.rand(m, generator=g, dtype=torch.float64, device="cuda"))
    G = torch.randn(n, 8, generator=g, dtype=torch.float64, device="cuda")
    P0 = G @ G.T / n
    A, C = -torch.eye(n, dtype=torch.float64, device="cuda"), torch.ones(1, n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()                     # the plan works on a stream of its own
    plan = dme.Plan(A, C=C, h=0.1, flows=["F3"], comp="lie", B=B, R=R,
                    prec="split_bf16")
    P = P0.clone()
    torch.cuda.synchronize()
    plan.apply("F3", 0.1, P)
    Z = P0 @ B
    ref = P0 - 0.1 * Z @ torch.linalg.solve(R + 0.1 * B.T @ Z, Z.T)
    assert (torch.linalg.norm(P - ref) / torch.linalg.norm(ref)).item() < SPLIT_TOL
    assert torch.equal(P, P.T)


# split-precision products in 128, 64 and 32 wide tiles (the width follows from the number of
# tiles), whole and cut at the right and lower edges, odd and even multiples of 32 along K
@pytest.mark.parametrize("pairs", [10, 13, 14])
@pytest.mark.parametrize("n", [31, 33, 63, 65, 96, 127, 129, 161, 289, 385, 545, 800])
def test_split_tile_widths_match_oracle(n, pairs):
    r = np.random.default_rng(n)
    A, C, S = _stable(n, n), r.standard_normal((2, n)), 0.1 * r.standard_normal((n, n)) / np.sqrt(n)
    P0 = W.random_psd(n, 4)
    plan = dme.Plan(dev(A), C=dev(C), h=0.05, flows=["F12", "F4"], S=dev(S), prec="split_bf16", pairs=pairs)
    ref = O.Plan(A, C.T @ C, None, None, S)
    for flow in ("F12", "F4"):
        P = dev(P0)
        plan.apply(flow, 0.05, P)
        assert rel(host(P), ref.apply(flow, 0.05, P0, "midpoint")) < SPLIT_TOL
        assert torch.equal(P, P.T)


# grouped launches: rows on both sides of the block-per-row slicing (K = 129) and of the narrow
# tiles, alone in the queue and together
@pytest.mark.parametrize("prec,tol", [("split_bf16", SPLIT_TOL), ("fp64", FP64_TOL)])
def test_served_sizes_match_their_own_plans(prec, tol):
    sizes = [1, 33, 97, 128, 129, 200, 257, 385]
    srv = dme.dme_server_create(4 << 30, 16)
    try:
        jobs = []
        for n in sizes:
            r = np.random.default_rng(n)
            m = 1 + n % 8
            A, C, B = _stable(n, n), r.standard_normal((2, n)), r.standard_normal((n, m))
            P0 = W.random_psd(n, 6)
            jobs.append((n, m, A, C, B, np.diag(0.5 + r.uniform(size=m)), P0))
        out = {}
        for together in (False, True):
            tickets = []
            for n, m, A, C, B, R, P0 in jobs:
                d = dme.make_desc(n, m=m, p=2, eq=dme.DME_DRE, comp="strang", flows=["F12", "F3"], prec=prec, h=0.02,
                                  q_is_factor=True)
                t = dme.dme_submit(srv, d, A, C, B, R, None, P0, 0.1, 5)
                if together:
                    tickets.append(t)
                else:
                    out[n] = np.empty((n, n))
                    dme.dme_poll(srv, t, out[n])
            for (n, m, A, C, B, R, P0), t in zip(jobs, tickets):
                P = np.empty((n, n))
                dme.dme_poll(srv, t, P)
                assert np.array_equal(P, out[n])
        for n, m, A, C, B, R, P0 in jobs:
            plan = dme.Plan(dev(A), C=dev(C), h=0.02, flows=["F12", "F3"], B=dev(B), R=dev(R))
            P = torch.empty(n, n, dtype=torch.float64, device="cuda")
            plan.solve(dev(P0), 0.1, 5, P)
            assert rel(out[n], host(P)) < tol
    finally:
        dme.dme_server_destroy(srv)


# the factored compressions: few and many columns at once (warp and block edges of the
# pivoted factorisations, a root of T3 beside them), a state that is zero, repeated columns
@pytest.mark.parametrize("p,m", [(1, 1), (2, 8), (15, 3), (31, 1), (33, 9)])
@pytest.mark.parametrize("prec,tol", [("fp64", FP64_TOL), ("split_bf16", SPLIT_TOL)])
def test_factored_ranks_match_dense_schemes(p, m, prec, tol):
    n = 230
    r = np.random.default_rng(p)
    A, B, R = _stable(n, p) / 2, r.standard_normal((n, m)) / np.sqrt(n), np.eye(m)
    C = r.standard_normal((p, n)) * np.exp2(-np.arange(p) % 12)[:, None]
    if p > 8:
        C[5] = C[2]
    flows = ["F1", "F2", "F3"]
    plan = dme.LowRankPlan(dev(A), dev(C), h=0.02, flows=flows, B=dev(B), R=dev(R), tol=1e-15, prec=prec)
    P = np.empty((n, n))
    plan.solve(0.1, 5, P_out=P)
    full = dme.Plan(dev(A), C=dev(C), h=0.02, flows=flows, B=dev(B), R=dev(R))
    ref = torch.empty(n, n, dtype=torch.float64, device="cuda")
    full.solve(np.zeros((n, n)), 0.1, 5, ref)
    assert rel(P, host(ref)) < tol


# columns beyond the capacity are refused, after the factor has been brought to its rank
@pytest.mark.parametrize("p,m,cols", [(64, 32, 233), (97, 2, 289)])
def test_factored_capacity_is_refused(p, m, cols):
    n = 230
    r = np.random.default_rng(p)
    A, B, R = _stable(n, p) / 2, r.standard_normal((n, m)) / np.sqrt(n), np.eye(m)
    C = r.standard_normal((p, n)) * np.exp2(-np.arange(p) % 12)[:, None]
    C[5] = C[2]
    plan = dme.LowRankPlan(dev(A), dev(C), h=0.02, flows=["F1", "F2", "F3"], B=dev(B), R=dev(R), tol=1e-15)
    with pytest.raises(dme.DmeError, match=f"{cols} columns exceed the capacity 224"):
        plan.solve(0.1, 5)


# ---- the Leja action, one T1 flow of a given factor
def _t1(A, L0, t):
    n = A.shape[0]
    plan = dme.LowRankPlan.from_csr(A, np.ones((1, n)), h=t, flows=["F1"], comp="lie", tol=1e-16, rmax=128)
    P = np.empty((n, n))
    plan.solve(t, 1, L0=L0, D0=np.eye(L0.shape[1]), P_out=P)
    return P


# stored entries on chip and not (a dense row), one and two entries per thread and more,
# symmetric (few substeps) and not (many), |t A| from far below one to several substeps.
# Bound: a substep adds at most (terms x stored entries per row) u relative to |L0|; ten of
# 80 terms and 8 entries are 1.5e-12, and P is a product of two.
@pytest.mark.parametrize("sym", [True, False])
@pytest.mark.parametrize("n,k,scale,dense_row", [(1, 1, 3.0, False), (2, 2, 1e-3, False), (7, 3, 10.0, False),
                                                 (255, 1, 30.0, False), (257, 5, 60.0, False), (300, 33, 20.0, True),
                                                 (600, 7, 2.0, True), (900, 64, 45.0, False)])
def test_leja_action_matches_dense_exponential(n, k, scale, dense_row, sym):
    r = np.random.default_rng(n)
    off = np.ones(max(n - 1, 0))
    A = sp.lil_matrix(sp.diags([off, -2.0 * np.ones(n), off * (1.0 if sym else 0.6)], [-1, 0, 1]))
    if dense_row:                      # an arrow: weak enough to leave the spectrum near [-4, 0]
        v = r.uniform(0.5, 1.0, n) / n
        A[0, :] = A[0, :] + v[None, :]
        if sym:
            A[:, 0] = A[:, 0] + v[:, None]
    A = sp.csr_matrix(A) * scale
    L0 = r.standard_normal((n, k))
    P = _t1(A, L0, 1.0)
    EL = scipy.linalg.expm(A.T.toarray()) @ L0
    assert np.linalg.norm(P - EL @ EL.T) <= 3e-12 * np.linalg.norm(L0 @ L0.T, 2) * np.sqrt(n)


# several thousand rows: two entries per thread on chip (n k = 256000) and more (512000)
@pytest.mark.parametrize("n,k", [(4000, 64), (8000, 64)])
def test_leja_action_of_large_blocks_matches_sine_transform(n, k):
    off = np.ones(n - 1)
    t = 9.0
    A = sp.csr_matrix(sp.diags([off, -2.0 * np.ones(n), off], [-1, 0, 1])) * t
    L0 = np.random.default_rng(n).standard_normal((n, k))
    P = _t1(A, L0, 1.0)
    lam = t * (-2.0 + 2.0 * np.cos(np.pi * np.arange(1, n + 1) / (n + 1)))
    EL = scipy.fft.idst(np.exp(lam)[:, None] * scipy.fft.dst(L0, 1, axis=0, norm="ortho"), 1, axis=0, norm="ortho")
    X = np.random.default_rng(1).standard_normal((n, 4))
    assert np.linalg.norm(P @ X - EL @ (EL.T @ X)) <= 3e-12 * np.linalg.norm(L0, 2) ** 2 * np.linalg.norm(X)


# a symmetric A is recognised in any stored order, and one that only its values make
# unsymmetric is not; entries stored twice are added either way
@pytest.mark.parametrize("form", ["sorted", "reversed", "twice", "perturbed"])
def test_leja_action_of_stored_orders(form):
    n, k, t = 130, 6, 25.0
    off = np.ones(n - 1)
    A = sp.csr_matrix(sp.diags([off, -2.0 * np.ones(n), off], [-1, 0, 1])) * t
    if form == "perturbed":
        A[3, 4] = 0.5 * t
    cols = [list(A.indices[A.indptr[i]:A.indptr[i + 1]]) for i in range(n)]
    vals = [list(A.data[A.indptr[i]:A.indptr[i + 1]]) for i in range(n)]
    if form == "reversed":
        cols, vals = [c[::-1] for c in cols], [v[::-1] for v in vals]
    if form == "twice":
        cols, vals = [c + c[:1] for c in cols], [[0.5 * v[0]] + v[1:] + [0.5 * v[0]] for v in vals]

    class Csr:
        shape = (n, n)
        indptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int32)
        indices = np.concatenate(cols).astype(np.int32)
        data = np.concatenate(vals).astype(np.float64)

    L0 = np.random.default_rng(2).standard_normal((n, k))
    P = _t1(Csr(), L0, 1.0)
    EL = scipy.linalg.expm(A.T.toarray()) @ L0
    assert np.linalg.norm(P - EL @ EL.T) <= 3e-12 * np.linalg.norm(L0 @ L0.T, 2) * np.sqrt(n)
