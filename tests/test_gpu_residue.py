"""FP64 plans of n >= 192: the congruence G P G^T by exact residue products, against
quadruple-precision sums.  Every entry must be within the a-priori bound of two
chained FP64 products of length n, (2 n + 4) u |G| |P| |G|^T entrywise, whatever
the scaling of the rows: what the residues cannot certify is recomputed in FP64."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_1805_08990_gb300 as dme
from gpu_util import FP64_TOL, dev, host, rel, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _gpu():
    require_gpu()


def _case(n, kind, seed):
    """A (its exponential is the operand) and a symmetric P."""
    r = np.random.default_rng(seed)
    A = r.standard_normal((n, n)) / np.sqrt(n) - 2.0 * np.eye(n)
    G = r.standard_normal((n, 12))
    P = G @ G.T
    if kind == "decay":                # entries falling off to 1e-60 away from the diagonal
        k = np.arange(n)
        P = P * np.exp2(-np.abs(k[:, None] - k[None, :]) * (200.0 / n))
    elif kind == "units":              # two decoupled blocks in units 2^40 apart, P coupled
        m = n // 3
        A[:m, m:] = 0.0
        A[m:, :m] = 0.0
        d = np.where(np.arange(n) < m, 2.0 ** 20, 2.0 ** -20)
        P = d[:, None] * P * d[None, :]
    elif kind == "zeros":              # zero rows and columns, and a zero block of A
        P[n // 2:, :] = 0.0
        P[:, n // 2:] = 0.0
        A[: n // 4, n // 4:] = 0.0
    elif kind == "tiny":               # beyond the residues' exponent range
        P = P * 2.0 ** -450
    return A, 0.5 * (P + P.T)


@pytest.mark.parametrize("n,kind", [(192, "dense"), (193, "decay"), (255, "units"), (256, "dense"), (257, "zeros"),
                                    (385, "units"), (321, "tiny"), (1023, "decay"), (1024, "dense"), (1025, "units"),
                                    (1100, "dense"), (2049, "dense")])
def test_congruence_entrywise_bound(n, kind):
    A, P0 = _case(n, kind, n)
    t = 0.3
    plan = dme.Plan(dev(A), C=dev(np.ones((1, n))), h=t, flows=["F1", "F2"], comp="lie")
    E = torch.empty(n, n, dtype=torch.float64, device="cuda")
    plan.expm(t, E, None)
    P = dev(P0)
    plan.apply("F1", t, P)
    got, E = host(P), host(E)
    assert np.array_equal(got, got.T)
    rows = np.unique(np.concatenate([[0, 1, 127, 128, 191, n // 3 - 1, n // 3, n // 2, n - 2, n - 1],
                                     np.random.default_rng(1).integers(0, n, 6)])) if n > 400 else np.arange(0, n, 3)
    q = np.longdouble
    Eq, Pq = E.astype(q), P0.astype(q)
    X = Eq[:, rows].T @ Pq
    ref = X @ Eq
    S = (np.abs(E)[:, rows].T @ np.abs(P0)) @ np.abs(E)
    bound = (2 * n + 4) * 2.0 ** -53 * S
    err = np.abs((got[rows] - ref).astype(np.float64))
    assert np.all(err <= bound), (err / np.where(bound > 0, bound, 1)).max()
    if kind == "dense":                # and in norm no worse than FP64 sums in order
        nat = np.linalg.norm((P0 @ E).T[rows] @ E - ref.astype(np.float64)) / np.linalg.norm(ref.astype(np.float64))
        assert np.linalg.norm(err) / np.linalg.norm(ref.astype(np.float64)) <= max(4e-16, 2.0 * nat)


def test_non_finite_entries_travel_as_in_fp64():
    n = 200
    A, P0 = _case(n, "dense", 3)
    A[:100, 100:] = 0.0
    A[100:, :100] = 0.0
    plan = dme.Plan(dev(A), C=dev(np.ones((1, n))), h=0.3, flows=["F1", "F2"], comp="lie")
    P = dev(P0)
    P[7, 7] = float("nan")
    P[150, 150] = float("inf")
    plan.apply("F1", 0.3, P)
    got = host(P)
    assert np.isnan(got[:100, :100]).all()           # E has no zeros inside its blocks
    assert not np.isfinite(got[100:, 100:]).any()


def test_generalised_steps_match_fp64_sums():
    """T4 (midpoint and Euler) on residue products: alpha, two and three addends."""
    n = 300
    r = np.random.default_rng(5)
    A, P0 = _case(n, "dense", 4)
    S = r.standard_normal((n, n)) / np.sqrt(n)
    for rule in (dme.DME_T4_MIDPOINT, dme.DME_T4_EULER):
        plan = dme.Plan(dev(A), C=dev(np.ones((1, n))), h=0.25, flows=["F12", "F4"], comp="strang", S=dev(S), t4_rule=rule)
        P = dev(P0)
        plan.apply("F4", 0.25, P)
        q = np.longdouble
        X = S.astype(q) @ P0.astype(q) @ S.astype(q).T
        ref = P0 + 0.25 * X + (0.25 ** 2 / 2 * (S.astype(q) @ X @ S.astype(q).T) if rule == dme.DME_T4_MIDPOINT else 0)
        assert np.linalg.norm((host(P) - ref).astype(np.float64)) <= 1e-15 * np.linalg.norm(ref.astype(np.float64))


@pytest.mark.parametrize("n", [192, 257, 448])
@pytest.mark.parametrize("kind", ["dense", "rotation", "graded"])
def test_exponential_solves(n, kind):
    """The exponential's solves: refined from an FP32 inverse (dense), given up for the pivoted
    elimination where that inverse fails (rotation by pi: the leading blocks of the Pade
    denominator are singular, the matrix is not), and not tried for an unbalanced operator."""
    r = np.random.default_rng(n)
    if kind == "rotation":
        m = n // 2
        A = np.zeros((n, n))
        A[np.arange(m), m + np.arange(m)] = np.pi
        A[m + np.arange(m), np.arange(m)] = -np.pi
        ref = np.eye(n)
        ref[: 2 * m, : 2 * m] *= -1.0
        t = 1.0
    else:
        A = r.standard_normal((n, n)) / np.sqrt(n) - 2.0 * np.eye(n)
        t = 0.4
        ref = O.expm(t * A)
        if kind == "graded":
            d = np.exp2(np.linspace(-6.0, 6.0, n))
            A = A * d[None, :] / d[:, None]
    plan = dme.Plan(dev(A), C=dev(np.full((1, n), 1e-3)), h=t, flows=["F1", "F2"], comp="lie")
    E = torch.empty(n, n, dtype=torch.float64, device="cuda")
    plan.expm(t, E, None)
    got = host(E)
    if kind == "graded":
        got = got * d[:, None] / d[None, :]
    assert rel(got, ref) < FP64_TOL
