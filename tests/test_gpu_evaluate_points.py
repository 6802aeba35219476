"""Evaluation from one point to more than fill the GPU: the blocks that share a
group of points change with their number (clusters of two, four and eight blocks,
one block with all or with fewer points than lanes), the values do not.  Against
the oracle (bound 1e-12 sum |c|) and, bit for bit, point by point between the calls."""
import numpy as np
import pytest
import torch

import paper_2309_14584_gb300 as F
import workloads as W
from oracle import fct_oracle as O

pytestmark = pytest.mark.gpu

# supports of 6..64 chunks: 32 points per block (short tables), 16 and 8 (long or
# many axes), 4 (deep), tables that take longer than a chunk
SUPPORTS = {
    "D2_d13": lambda: W.total_degree_support(2, 13),
    "D3_d9": lambda: W.total_degree_support(3, 9),
    "D6_d5": lambda: W.total_degree_support(6, 5),
    "D8_d5": lambda: W.total_degree_support(8, 5),
    "D2_d150": lambda: W.total_degree_support(2, 150),
    "D1_d700": lambda: W.total_degree_support(1, 700),
    "sparse_d100": lambda: W.sparse_infinity_support(3, 100, 9, 3000, 3),
    "nz10": lambda: W.sparse_support_vectorised(3, 128, 2, 1500, 10),
    "nz45": lambda: W.sparse_support_vectorised(3, 128, 2, 1100, 45),
}


@pytest.mark.parametrize("name", SUPPORTS)
def test_values_do_not_depend_on_the_number_of_points(name):
    sup = SUPPORTS[name]()
    N, D = sup.shape
    plan = F.Plan(sup, np.full((1, D), 1, dtype=np.int32))
    g = W.stream(93, "probe")
    c = g.standard_normal(N)
    pts = g.uniform(-1.0, 1.0, (9800, D))
    cd, pd = torch.from_numpy(c).cuda(), torch.from_numpy(pts).cuda()
    ref = torch.full((9800,), float("nan"), dtype=torch.float64, device="cuda")
    plan.evaluate(cd, pd, ref)
    want = O.evaluate_expansion(c, sup, pts[:60])
    assert np.max(np.abs(ref[:60].cpu().numpy() - want)) <= 1e-12 * np.abs(c).sum()
    for P in (1, 2, 31, 33, 600, 1217, 1216, 2431, 2433, 4864, 4866, 7000, 9728):
        vals = torch.full((P + 1,), float("nan"), dtype=torch.float64, device="cuda")
        plan.evaluate(cd, pd[:P], vals[:P])
        torch.cuda.synchronize()
        assert torch.equal(vals[:P], ref[:P]) and torch.isnan(vals[P]), P
    plan.close()


def test_few_points_use_the_whole_gpu():
    # 32 points of a D = 6 degree 10 expansion against 304 times as many, which fill
    # the GPU: 0.10 of their time; by one block alone 0.21
    sup = W.total_degree_support(6, 10)
    plan = F.Plan(sup, np.full((1, 6), 1, dtype=np.int32))
    c = torch.ones(len(sup), dtype=torch.float64, device="cuda")
    t = {}
    for P in (32, 32 * 304):
        pts = torch.rand(P, 6, dtype=torch.float64, device="cuda") * 2 - 1
        vals = torch.empty(P, dtype=torch.float64, device="cuda")
        ms = []
        for _ in range(7):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(20):
                plan.evaluate(c, pts, vals)
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        t[P] = sorted(ms)[3]
    assert t[32] <= 0.15 * t[32 * 304], t
    plan.close()
