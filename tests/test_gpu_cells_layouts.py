"""The layouts that the inner solve by grid groups can take, each shown to be the one
that ran: one grid per group and several, one slice of coefficients and several, with
short last groups and slices, on both grid kinds (first-kind entries are signed), and
the FP64 solve that takes over from it.

The target is a polynomial on the support, so the coefficients are known.  A solve
that ends with |A^T r| <= tol |A^T b| is within tol kappa^2 of them; the estimate of
kappa is a lower bound, taken twice, and rounding is allowed 1e-11."""
import numpy as np
import pytest
import torch

import paper_2309_14584_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-12
# N, nonzeros, degree, D, K, block threads, grid kind, several grids per group?, several slices?
CASES = [
    (6145, 3, 4, 30, 331, 512, F.FCT_GRID_EXTREMA, True, False),
    (9001, 3, 9, 60, 335, 256, F.FCT_GRID_EXTREMA, True, False),
    (9001, 3, 9, 60, 335, 256, F.FCT_GRID_FIRST_KIND, True, False),
    (12001, 3, 5, 60, 305, 128, F.FCT_GRID_FIRST_KIND, False, False),
    (30001, 3, 3, 100, 400, 128, F.FCT_GRID_EXTREMA, False, True),
    (20001, 3, 9, 100, 1001, 128, F.FCT_GRID_EXTREMA, True, True),
    (20001, 3, 9, 100, 1001, 128, F.FCT_GRID_FIRST_KIND, True, True),
    (50001, 10, 3, 100, 241, 512, F.FCT_GRID_EXTREMA, True, True),
]


def _problem(N, nz, d, D, K):
    sup = W.sparse_infinity_support(13, D, d, N, nz) if nz == 3 and d == 9 else W.sparse_support_vectorised(3, D, d, N,
                                                                                                            nz)
    return sup, W.l_grid(700 + D, N, D, K, 1, d + 1), W.poly_coefficients(10, sup)


def _bound(plan):
    start = torch.from_numpy(W.stream(5, "probe").standard_normal(plan.N)).cuda()
    work = torch.empty(plan.N, dtype=torch.float64, device="cuda")
    kappa = F.fct_plan_condition(plan.handle, start, work, 400)["kappa"]
    return 4.0 * kappa ** 2 * TOL + 1e-11


def _solve(plan, c_true):
    x = torch.empty(plan.M, dtype=torch.float64, device="cuda")
    plan.sample(W.FAMILY_POLY | F.fct.FCT_SAMPLE_FOLDED, c_true, x)
    c = torch.full((plan.N,), float("nan"), dtype=torch.float64, device="cuda")
    rep = plan.execute(x, c)
    assert rep["status"] == 0, rep
    got = c.cpu().numpy()
    return rep, np.linalg.norm(got - c_true) / np.linalg.norm(c_true), got


@pytest.mark.parametrize("N,nz,d,D,K,bt,kind,groups,slices", CASES)
def test_layout_and_result(N, nz, d, D, K, bt, kind, groups, slices):
    sup, (sizes, nodes), c_true = _problem(N, nz, d, D, K)
    opts = dict(precision=F.FCT_MIXED, tol=TOL, inner_tol=1e-4, max_iter=20000, block_threads=bt, grid_kind=kind)
    plan = F.Plan(sup, sizes, nodes, **opts)
    lay = F.fct_plan_get_inner_layout(plan.handle)
    assert plan.info["kernel_variant"] == 3 and lay["groups"] == -(-K // lay["grids_per_group"])
    assert (lay["grids_per_group"] > 1, lay["slices"] > 1) == (groups, slices), lay
    assert (lay["slices"] - 1) * lay["slice_coefs"] < N < lay["slices"] * lay["slice_coefs"]  # the last is short
    rep, err, got = _solve(plan, c_true)
    assert rep["refinements"] > 1
    assert err <= _bound(plan), (err, _bound(plan))
    # the host-built tables give the same bits; a clone has the same layout
    host = F.Plan(sup, sizes, nodes, plan_build=F.FCT_PLAN_BUILD_HOST, **opts)
    assert F.fct_plan_get_inner_layout(host.handle) == lay
    assert np.array_equal(_solve(host, c_true)[2], got)
    host.close()
    clone = plan.clone()
    assert F.fct_plan_get_inner_layout(clone.handle) == lay
    clone.close()
    plan.close()


def test_fp64_takes_over_after_one_sweep():
    sup, (sizes, nodes), c_true = _problem(9001, 3, 9, 60, 335)
    plan = F.Plan(sup, sizes, nodes, precision=F.FCT_MIXED, tol=TOL, inner_tol=1e-4, max_refine=1)
    assert plan.info["kernel_variant"] == 3
    rep, err, _ = _solve(plan, c_true)
    assert rep["refinements"] == 1
    assert err <= _bound(plan)
    plan.close()


def test_other_plans_report_no_layout():
    sup, (sizes, nodes), _ = _problem(6145, 3, 4, 30, 331)
    none = {"groups": 0, "grids_per_group": 0, "slices": 0, "slice_coefs": 0}
    # FP64, too few grids, too few coefficients
    for plan in (F.Plan(sup, sizes, nodes),
                 F.Plan(sup, sizes[:150], nodes[:150], precision=F.FCT_MIXED, tol=TOL, inner_tol=1e-4),
                 F.Plan(sup[:6143], sizes, nodes, precision=F.FCT_MIXED, tol=TOL, inner_tol=1e-4)):
        assert F.fct_plan_get_inner_layout(plan.handle) == none and plan.info["kernel_variant"] != 3
        plan.close()
