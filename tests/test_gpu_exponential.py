"""E_t of FP64 plans of n >= 192 against Kronecker products of extended-precision exponentials:
A = I x T + T x I has e^{tA} = e^{tT} x e^{tT}.  A balanced A's powers, squarings and refined
solves run without certificates and are normwise accurate: an error of 64 u in the largest
Pade form (|tA| <= 5.4), doubled by each of the s squarings."""
import math

import numpy as np
import pytest
import torch

import paper_1805_08990_gb300 as dme
from gpu_util import dev, host, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _gpu():
    require_gpu()


def _factor(kind, nx):
    one = np.ones(nx - 1)
    T = np.diag(one, -1) - 2.0 * np.eye(nx) + np.diag(one, 1)
    if kind == "convection":
        T = T - 0.3 * (np.diag(one, 1) - np.diag(one, -1))
    elif kind == "dense":
        T = np.random.default_rng(nx).standard_normal((nx, nx)) / np.sqrt(nx) - 2.0 * np.eye(nx)
    elif kind == "graded":             # row and column sums 2^12 apart: pivoted elimination, certified products
        d = np.exp2(np.linspace(-3.0, 3.0, nx))
        T = T * d[None, :] / d[:, None]
    return T


@pytest.mark.parametrize("kind", ["heat", "convection", "dense", "graded"])
@pytest.mark.parametrize("nx,norm", [(14, 0.3), (17, 5.0), (17, 40.0), (23, 5.0)])
def test_kronecker_sum(kind, nx, norm):
    T = _factor(kind, nx)
    one = np.eye(nx)
    A = np.kron(one, T) + np.kron(T, one)
    n = nx * nx
    t = norm / np.abs(A).sum(0).max()
    q = np.longdouble
    X = T.astype(q) * q(t) / 1024
    e = np.eye(nx, dtype=q)
    term = e.copy()
    for j in range(1, 20):
        term = term @ X / j
        e = e + term
    for _ in range(10):
        e = e @ e
    plan = dme.Plan(dev(A), C=dev(np.full((1, n), 1e-3)), h=t, flows=["F1", "F2"], comp="lie")
    E = torch.empty(n, n, dtype=torch.float64, device="cuda")
    plan.expm(t, E, None)
    ref = np.kron(e, e)
    err = float(np.linalg.norm((host(E) - ref).astype(np.float64)) / np.linalg.norm(ref.astype(np.float64)))
    s = max(0, math.ceil(math.log2(1.01 * norm / 5.37)))
    assert err <= 64 * 2.0 ** s * 2.0 ** -53
