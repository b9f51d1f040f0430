"""FP64 products whose residue sums are as large as they get: rows of one constant, so that
every term of a sum has the same residue and sign."""
import numpy as np
import pytest
import torch

import paper_1805_08990_gb300 as dme
from gpu_util import dev, host, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _gpu():
    require_gpu()


# (n, a, b): n a b has a residue sum near -2^24 modulo 255 in integers of 61 - log2 |row| bits
CASES = [(577, 0.8251856099188752, 0.358081198534387), (577, -0.6743668325837577, 0.6942725357276607),
         (853, 0.6257815933973978, 0.7864648019957695), (853, -0.10328771224131583, 0.3026237893873138),
         (1021, 0.4778152288085107, 0.6773822806304568), (1021, -0.7731704195343296, 0.1677869334346773),
         (1024, -0.31116594213485516, 0.37246532836315493), (1024, -0.8688898331736545, 0.9979833558848721),
         (1024, 0.9051924950571193, 0.873609794533183), (1024, 0.25091920048512395, 0.6978108688532659)]


@pytest.mark.parametrize("n,a,b", CASES)
def test_constant_rows(n, a, b):
    """T4 (Euler) with S = a 1 1^T on P = b 1 1^T: every entry is b + t n^2 a^2 b, each of the two
    products within K u of its sum."""
    t = 0.25
    A = -np.eye(n)
    plan = dme.Plan(dev(A), C=dev(np.ones((1, n))), h=t, flows=["F12", "F4"], comp="lie", S=dev(np.full((n, n), a)),
                    t4_rule=dme.DME_T4_EULER)
    P = dev(np.full((n, n), b))
    torch.cuda.synchronize()
    plan.apply("F4", t, P)
    want = b + t * n * n * a * a * b
    assert np.abs(host(P) - want).max() <= (2 * n + 8) * 2.0 ** -53 * abs(want)


@pytest.mark.parametrize("n", [192, 1025])
def test_products_of_subnormal_entries(n):
    """An output whose only nonzero product has a subnormal factor is that product: S P S^T with
    S[i, k] = 2^-1060 beside an entry 1, P = 2^390 e_k e_k^T."""
    i, j, k = n // 3, n - 2, n // 2
    S = np.zeros((n, n))
    S[i, 5] = S[j, k] = 1.0
    S[i, k] = 2.0 ** -1060
    P0 = np.zeros((n, n))
    P0[k, k] = 2.0 ** 390
    plan = dme.Plan(dev(-np.eye(n)), C=dev(np.ones((1, n))), h=0.5, flows=["F12", "F4"], comp="lie", S=dev(S),
                    t4_rule=dme.DME_T4_EULER)
    P = dev(P0)
    torch.cuda.synchronize()
    plan.apply("F4", 0.5, P)
    want = P0.copy()
    want[j, j] += 0.5 * 2.0 ** 390
    want[i, j] = want[j, i] = 0.5 * 2.0 ** -670
    assert np.array_equal(host(P), want)


@pytest.mark.parametrize("n", [192, 231, 416])
@pytest.mark.parametrize("c", [1, 7, 8, 9, 32])
def test_outputs_without_certificate(n, c):
    """c columns of each 32 of P have no entry where the rows of S are large, so that 8 c of a
    strip's 256 outputs fail the certificate (recomputed one by one up to 64, as a strip
    beyond).  Bound: two chained FP64 products of length n, entrywise."""
    r = np.random.default_rng(n + c)
    S = r.standard_normal((n, n)) * 2.0 ** -30
    S[:, 0] = 1.0
    G = r.standard_normal((n, 8))
    P0 = G @ G.T + 3.0
    J = np.arange(n) % 32 >= 32 - c
    J[0] = False
    P0[0, J] = P0[J, 0] = 0.0
    t = 0.5
    plan = dme.Plan(dev(-np.eye(n)), C=dev(np.ones((1, n))), h=t, flows=["F12", "F4"], comp="lie", S=dev(S),
                    t4_rule=dme.DME_T4_EULER)
    P = dev(P0)
    torch.cuda.synchronize()
    plan.apply("F4", t, P)
    got = host(P)
    assert np.array_equal(got, got.T)
    q = np.longdouble
    rows = np.arange(0, n, 5)
    ref = P0[rows] + t * ((S[rows].astype(q) @ P0.astype(q)) @ S.T.astype(q))
    mag = np.abs(P0[rows]) + t * ((np.abs(S[rows]) @ np.abs(P0)) @ np.abs(S.T))
    err = np.abs((got[rows] - ref).astype(np.float64))
    assert np.all(err <= (2 * n + 6) * 2.0 ** -53 * mag)
