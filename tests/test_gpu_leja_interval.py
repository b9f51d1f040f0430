"""The Leja action of symmetric operators whose spectrum ends short of their Gershgorin
interval: e^{tA} L0 (L0's columns: ones, random, a unit vector) against a Taylor sum in
extended precision, beside the oracle's action (substeps of t g <= 4, float64)."""
import numpy as np
import pytest
import scipy.sparse as sp

import paper_1805_08990_gb300 as dme
from gpu_util import require_gpu
from oracle import dme_leja

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _gpu():
    require_gpu()


def _operator(kind):
    nx = 14
    l1 = sp.diags([np.ones(nx - 1), -2.0 * np.ones(nx), np.ones(nx - 1)], [-1, 0, 1])
    L = sp.kron(sp.eye(nx), l1) + sp.kron(l1, sp.eye(nx))
    r = np.random.default_rng(0)
    if kind == "heat":                 # 2 - x = 0.04
        return L
    if kind == "signs":                # the same spectrum, D L D with signs D
        D = sp.diags(np.sign(r.standard_normal(nx * nx)))
        return D @ L @ D
    if kind == "biharmonic":           # 1.1
        return -(L @ L)
    S = np.triu((r.random((200, 200)) < 0.08) * r.choice([-1.0, 1.0], (200, 200)), 1)   # random signs: 1.4
    S = S + S.T
    return sp.csr_matrix(S - np.abs(S).sum(1).max() * np.eye(200))


def _exact(A, V, t):
    q = np.longdouble
    A, V = A.astype(q), V.astype(q)
    k = max(1, int(np.ceil(0.5 * t * float(np.abs(A).sum(1).max()))))     # |A| t / k <= 2
    for _ in range(k):
        term = V.copy()
        for j in range(1, 32):
            term = A @ term * (q(t) / k / j)
            V = V + term
    return V


@pytest.mark.parametrize("tg", [9.9, 18.6])
@pytest.mark.parametrize("kind", ["heat", "signs", "biharmonic", "random"])
def test_action_is_as_accurate_as_short_substeps(kind, tg):
    A = sp.csr_matrix(_operator(kind))
    n = A.shape[0]
    lo, hi = dme_leja.gershgorin_interval(A)
    t = tg / (0.25 * (hi - lo))
    L0 = np.stack([np.ones(n), np.random.default_rng(1).standard_normal(n), np.eye(n)[n // 2]], 1)
    P = np.empty((n, n))
    plan = dme.LowRankPlan.from_csr(A, np.ones((1, n)), h=t, flows=["F1"], comp="lie", tol=1e-16)
    plan.solve(t, 1, L0=L0, D0=np.eye(3), P_out=P)
    V = _exact(A.toarray(), L0, t)
    ref = V @ V.T
    W = dme_leja.leja_action(A.T.tocsr(), L0, t)
    err = lambda X: float(np.linalg.norm((X - ref).astype(np.float64)) / np.linalg.norm(ref.astype(np.float64)))  # noqa: E731
    # the same method in the same precision: a few times the oracle's error, or of 40 terms' rounding
    assert err(P) <= 8.0 * max(err(W @ W.T), 40 * 2.0 ** -53)
