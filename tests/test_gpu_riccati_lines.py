"""T3 on both sides of its kernels' lines: rows per block, Y inside the update or beside it, the
partial Gram sums in one block or over the chip (m > 8), alone and in served groups."""
import numpy as np
import pytest
import torch

import paper_1805_08990_gb300 as dme
from gpu_util import FP64_TOL, dev, host, rel, require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True, scope="module")
def _gpu():
    require_gpu()


@pytest.mark.parametrize("n,m", [(1699, 5), (1700, 5), (1703, 8), (1705, 12), (1699, 32), (1700, 32), (833, 8), (834, 8),
                                 (1290, 5), (1291, 5), (1581, 4), (1582, 4)])
def test_flow_matches_formula(n, m):
    r = np.random.default_rng(n + m)
    B, R = r.standard_normal((n, m)), np.diag(0.5 + r.uniform(size=m))
    G = r.standard_normal((n, 8))
    P0 = G @ G.T / n
    plan = dme.Plan(dev(-np.eye(n)), C=dev(np.ones((1, n))), h=0.1, flows=["F3"], comp="lie", B=dev(B), R=dev(R))
    P = dev(P0)
    torch.cuda.synchronize()
    plan.apply("F3", 0.1, P)
    Z = P0 @ B
    ref = P0 - 0.1 * Z @ np.linalg.solve(R + 0.1 * B.T @ Z, Z.T)
    assert rel(host(P), ref) < FP64_TOL
    assert torch.equal(P, P.T)


def test_served_groups_of_many_inputs_equal_their_plans():
    srv = dme.dme_server_create(4 << 30, 16)
    try:
        jobs = []
        for n, m in ((40, 9), (65, 32), (90, 3), (120, 17), (150, 8), (160, 16)):
            r = np.random.default_rng(n)
            A = r.standard_normal((n, n)) / np.sqrt(n) - 2.5 * np.eye(n)
            B, C = r.standard_normal((n, m)), r.standard_normal((2, n))
            R, P0 = np.diag(0.5 + r.uniform(size=m)), np.zeros((n, n))
            d = dme.make_desc(n, m=m, p=2, eq=dme.DME_DRE, comp="strang", flows=["F12", "F3"], prec="fp64", h=0.02,
                              q_is_factor=True)
            jobs.append((n, A, B, C, R, P0, dme.dme_submit(srv, d, A, C, B, R, None, P0, 0.1, 5)))
        for n, A, B, C, R, P0, ticket in jobs:
            got, want = np.empty((n, n)), np.empty((n, n))
            dme.dme_poll(srv, ticket, got)
            plan = dme.Plan(dev(A), C=dev(C), h=0.02, flows=["F12", "F3"], B=dev(B), R=dev(R))
            plan.solve(P0, 0.1, 5, want)
            assert np.array_equal(got, want)
    finally:
        dme.dme_server_destroy(srv)
