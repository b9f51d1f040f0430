"""Plans of n >= 192 in a device with little free memory: the residue planes are held only while
they fit, and make room for what the plan cannot do without."""
import numpy as np
import pytest
import torch

import paper_1805_08990_gb300 as dme
from gpu_util import dev, host, rel, require_gpu

pytestmark = pytest.mark.gpu
MB = 1 << 20
N = 2048


@pytest.fixture(autouse=True, scope="module")
def _gpu():
    require_gpu()


def _data(n):
    r = np.random.default_rng(n)
    return (dev(r.standard_normal((n, n)) / np.sqrt(n) - 2.0 * np.eye(n)), dev(r.standard_normal((2, n))),
            dev(r.standard_normal((n, n)) / np.sqrt(n)))


def _run(kind, A, C, S):
    n = A.shape[0]
    if kind == "factored":
        plan = dme.LowRankPlan(A, C, h=0.1, flows=["F12"], comp="lie")
        plan.solve(0.2, 2)
        L, d = plan.factors()
        plan.close()
        return (L * d) @ L.T
    gen = kind == "generalised"
    plan = dme.Plan(A, C=C, h=0.1, flows=["F12", "F4"] if gen else ["F12"], comp="lie", S=S if gen else None)
    P = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    plan.step(P, 2)
    if kind == "lengths":              # E and W of six more step lengths stay in the plan
        for k in range(6):
            plan.apply("F12", 0.1 + 0.01 * k, P)
        plan.step(P, 1)
    torch.cuda.synchronize()
    plan.close()
    return host(P)


# 80 to 100 MB more than these plans need without planes (741, 851, 1103 and 1213 MB)
@pytest.mark.parametrize("kind,free_mb", [("dense", 840), ("generalised", 930), ("lengths", 1190), ("factored", 1310)])
def test_plan_fits_without_planes(kind, free_mb):
    small = _data(256)
    _run(kind, *small)                 # kernels loaded, pools warm
    full = _data(N)
    want = _run(kind, *full)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - free_mb * MB, dtype=torch.uint8, device="cuda")
    try:
        got = _run(kind, *full)
    finally:
        del fill
        torch.cuda.empty_cache()
    assert rel(got, want) < 1e-12


def test_plan_bytes_count_the_planes():
    """dme_plan_bytes: A, Q, X, E_t, W_t and, beside them, 34 bytes an entry for the planes of
    E_t^T and of the step operand and 17 for the workspace; less once they have made room."""
    n = N
    A, C, _ = _data(n)
    plan = dme.Plan(A, C=C, h=0.1, flows=["F12"], comp="lie")
    full = dme.dme_plan_bytes(plan.handle)
    assert (5 * 8 + 2 * 34 + 17) * n * n <= full <= (5 * 8 + 2 * 34 + 17) * n * n * 1.05
    plan.apply("F12", 0.1, torch.zeros(n, n, dtype=torch.float64, device="cuda"))
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - 500 * MB, dtype=torch.uint8, device="cuda")
    P = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    try:
        plan.apply("F12", 0.2, P)      # another E_t and W_t: 20 blocks of 32 MB beside the planes' 11
    finally:
        del fill
        torch.cuda.empty_cache()
    held = dme.dme_plan_bytes(plan.handle)
    assert 7 * 8 * n * n <= held <= 7 * 8 * n * n * 1.05
    plan.close()
