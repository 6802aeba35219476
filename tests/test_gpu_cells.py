"""The mixed path's inner solve by grid groups (plans with at least as many grids
as SMs and enough coefficients): one slice and several, one grid per group and
several, rows of one entry up to most columns of a grid, the three block sizes.
The target is a polynomial on the support, so the coefficients are known; the
bound is the mixed path's, 1e-10."""
import numpy as np
import pytest
import torch

import paper_2309_14584_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu

# N, nonzeros, degree, D, K, block threads: the smallest N that takes the path
# (6144) and a ragged one; K = 152 (one grid per group) to 330 (several, the last
# group short); N = 24001 (several slices at 128 and 256 threads); short rows
# (10 nonzero components) and rows of most columns (3)
CASES = [
    (6144, 10, 3, 30, 176, 256),
    (6145, 3, 4, 30, 330, 512),
    (7001, 10, 3, 40, 309, 256),
    (9999, 10, 3, 30, 176, 128),
    (24001, 10, 3, 60, 200, 256),
    (24001, 10, 3, 60, 153, 512),
]


@pytest.mark.parametrize("N,nz,d,D,K,bt", CASES)
def test_recovers_the_polynomial_whatever_the_builder_and_the_team(N, nz, d, D, K, bt):
    sup = W.sparse_support_vectorised(3, D, d, N, nz)
    sizes, nodes = W.l_grid(700 + D, N, D, K, 1, d + 1)
    c_true = W.poly_coefficients(10, sup)
    opts = dict(precision=F.FCT_MIXED, tol=1e-13, inner_tol=1e-5, block_threads=bt)
    plan = F.Plan(sup, sizes, nodes, **opts)
    host = F.Plan(sup, sizes, nodes, plan_build=F.FCT_PLAN_BUILD_HOST, **opts)
    x = torch.empty(plan.M, dtype=torch.float64, device="cuda")
    plan.sample(W.FAMILY_POLY | F.fct.FCT_SAMPLE_FOLDED, c_true, x)
    c = torch.full((N,), float("nan"), dtype=torch.float64, device="cuda")
    rep = plan.execute(x, c)
    assert rep["status"] == 0 and rep["refinements"] > 0, rep
    got = c.cpu().numpy()
    assert np.linalg.norm(got - c_true) / np.linalg.norm(c_true) <= 1e-10
    # the host-built tables and teams of other sizes give the same bits
    o = torch.full_like(c, float("nan"))
    assert host.execute(x, o)["iterations"] == rep["iterations"]
    assert torch.equal(o, c)
    clones = [plan.clone() for _ in range(2)]
    outs = [torch.full_like(c, float("nan")) for _ in clones]
    for team in (7, 76):
        reps = F.fct_execute_batch([p.handle for p in clones], [x] * 2, outs, team_blocks=team)
        assert all(r["status"] == 0 for r in reps)
        for o in outs:
            assert torch.equal(o, c)
    for p in clones + [host, plan]:
        p.close()


def test_nonfinite_samples_and_iteration_caps_are_reported():
    N, D = 6200, 30
    sup = W.sparse_support_vectorised(3, D, 3, N, 10)
    sizes, nodes = W.l_grid(730, N, D, 180, 1, 4)
    plan = F.Plan(sup, sizes, nodes, precision=F.FCT_MIXED, tol=1e-12, inner_tol=1e-4, max_iter=3, max_refine=1)
    x = torch.empty(plan.M, dtype=torch.float64, device="cuda")
    plan.sample(W.FAMILY_POLY | F.fct.FCT_SAMPLE_FOLDED, W.poly_coefficients(1, sup), x)
    c = torch.empty(N, dtype=torch.float64, device="cuda")
    with pytest.raises(F.FctError) as e:
        plan.execute(x, c)
    assert e.value.status == F.fct.FCT_ERR_NOCONV
    x[17] = float("nan")
    with pytest.raises(F.FctError) as e:
        plan.execute(x, c)
    assert e.value.status == F.fct.FCT_ERR_NONFINITE
    plan.close()
