"""Which solver kernel a launch takes: the variant with the inner solve by grid
groups only where a plan of the launch solves so (alone, without allocations, in a
batch; a server takes plans of either kind at any time), and a transform's
coefficients the same bit for bit in all of them."""
import numpy as np
import pytest
import torch

import paper_2309_14584_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu

CELLS = 3  # fct_plan_info.kernel_variant of plans whose inner solve runs by grid groups


def _cells_plan(bt=256, precision=None):
    N, D = 6200, 30
    sup = W.sparse_support_vectorised(3, D, 3, N, 10)
    sizes, nodes = W.l_grid(730, N, D, 180, 1, 4)
    return F.Plan(sup, sizes, nodes, precision=F.FCT_MIXED if precision is None else precision, tol=1e-12,
                  inner_tol=1e-4, block_threads=bt)


def _plain_plan(bt=256):
    w = W.make_workload("s6", 76, 6, 6, 18, 1, 7, W.FAMILY_GAUSSCOS, tol=1e-12, precision="mixed")
    return F.Plan(w.support, w.sizes, w.nodes, precision=F.FCT_MIXED, tol=1e-12, inner_tol=1e-4, block_threads=bt)


def _samples(plan, seed):
    x = torch.empty(plan.M, dtype=torch.float64, device="cuda")
    plan.sample(W.FAMILY_GAUSSCOS, W.gausscos_params(seed, plan.info["D"]), x)
    return x


def _nan(n):
    return torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("bt", [128, 256, 512])
def test_variant_of_single_launches_and_batches(bt):
    cells, plain = _cells_plan(bt), _plain_plan(bt)
    assert cells.info["kernel_variant"] == CELLS and plain.info["kernel_variant"] != CELLS
    f64 = _cells_plan(bt, F.FCT_FP64)
    assert f64.info["kernel_variant"] != CELLS
    f64.close()
    plans = [plain, cells, plain.clone(), cells.clone()]
    assert plans[3].info["kernel_variant"] == CELLS
    xs = [_samples(p, 5 + i) for i, p in enumerate(plans)]
    alone = []
    for p, x in zip(plans, xs):
        o = _nan(p.N)
        assert p.execute(x, o)["status"] == 0
        alone.append(o)
    # batches with and without plans that solve by grid groups, in either order
    for pick in ([0, 1, 2, 3], [3, 2], [0, 2]):
        for team in (0, 19):
            outs = [_nan(plans[i].N) for i in pick]
            reps = F.fct_execute_batch([plans[i].handle for i in pick], [xs[i] for i in pick], outs, team_blocks=team)
            assert all(r["status"] == 0 for r in reps)
            for i, o in zip(pick, outs):
                assert torch.equal(o, alone[i])
    # the condition estimate of a plan that solves by grid groups (FP64 on its tables)
    est = []
    for p in (cells, plans[3]):
        start = torch.from_numpy(W.stream(4, "probe").standard_normal(p.N)).cuda()
        est.append(F.fct_plan_condition(p.handle, start, _nan(p.N), 60)["kappa"])
    assert est[0] == est[1] and np.isfinite(est[0]) and est[0] > 1.0
    for p in plans[:1:-1] + [cells, plain]:
        p.close()


def test_without_allocations():
    """The fixed array holds a plan of 176 grids only with fewer points per grid than
    coefficients (about 3000 here)."""
    N, D = 6144, 30
    sup = W.sparse_support_vectorised(3, D, 3, N, 10)
    sizes, nodes = W.l_grid(730, 3000, D, 176, 1, 4)
    plan = F.Plan(sup, sizes, nodes, precision=F.FCT_MIXED, tol=1e-12, inner_tol=1e-4)
    assert plan.info["kernel_variant"] == CELLS
    x = _samples(plan, 3)
    alone, o = _nan(N), _nan(N)
    assert plan.execute(x, alone)["status"] == 0
    assert F.fct_execute_noalloc(plan.handle, x, o)["status"] == 0
    assert torch.equal(o, alone)
    plan.close()


def test_server_takes_plans_by_grid_groups_after_others():
    """The jobs before, beside and after the first one that solves by grid groups
    all finish, with the coefficients of a launch of their own."""
    cells, plain = _cells_plan(), _plain_plan()
    plans = [plain, plain.clone(), cells, cells.clone(), plain.clone()]
    xs = [_samples(p, 40 + i) for i, p in enumerate(plans)]
    alone = []
    for p, x in zip(plans, xs):
        o = _nan(p.N)
        assert p.execute(x, o)["status"] == 0
        alone.append(o)
    torch.cuda.synchronize()
    s = F.fct_server_create(256, 16, 0, 0.2)
    for order in ([0, 1], [0, 2, 1, 3, 4], [1, 3, 0]):
        for _ in range(3):
            outs = [_nan(plans[i].N) for i in order]
            torch.cuda.synchronize()
            tickets = [F.fct_server_submit(s, plans[i].handle, xs[i], o) for i, o in zip(order, outs)]
            for t in tickets:
                assert F.fct_server_wait(s, t, 60.0)["status"] == 0
            for i, o in zip(order, outs):
                assert torch.equal(o, alone[i])
    F.fct_server_destroy(s)
    for p in plans[::-1]:
        p.close()
