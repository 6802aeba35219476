"""Evaluation by shared prefixes at the sizes where its split can go wrong: one
term, the edges of its term chunks (N = 31, 32, 65, 1023, 1024), one point to a
few blocks, unordered supports, and tables that leave few points per block.  The
bound is 1e-12 sum |c|, as for the term-by-term kernel (a sum of N terms of
magnitude at most |c| in any order, each a product of at most D rounded factors
that a recurrence of at most d steps makes)."""
import numpy as np
import pytest
import torch

import paper_2309_14584_gb300 as F
import workloads as W
from oracle import fct_oracle as O

pytestmark = pytest.mark.gpu


def _shuffled(D, d, N):
    sup = W.total_degree_support(D, d)
    order = W.stream(7, "probe").permutation(len(sup))[:N]
    return np.ascontiguousarray(sup[order])


CASES = [
    ("one_term", lambda: np.zeros((1, 3), np.uint16), 5),
    ("n31", lambda: W.total_degree_support(3, 6)[:31], 33),
    ("n32_unordered", lambda: _shuffled(3, 6, 32), 32),
    ("n65", lambda: W.total_degree_support(4, 4)[:65], 31),
    ("n1023_unordered", lambda: _shuffled(5, 9, 1023), 1),
    ("n1024", lambda: W.total_degree_support(6, 8)[:1024], 700),
    ("sparse_d100", lambda: W.sparse_infinity_support(3, 100, 9, 3000, 3), 65),
    ("long_axis", lambda: W.total_degree_support(1, 700), 40),
    ("deep", lambda: np.ascontiguousarray(np.tri(60, 60, dtype=np.uint16)), 40),
]


@pytest.mark.parametrize("mk,P", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_matches_the_oracle_and_does_not_depend_on_the_other_points(mk, P):
    sup = mk()
    N, D = sup.shape
    plan = F.Plan(sup, np.full((1, D), 1, dtype=np.int32))
    g = W.stream(91, "probe")
    c = g.standard_normal(N)
    pts = g.uniform(-1.0, 1.0, (P, D))
    cd, pd = torch.from_numpy(c).cuda(), torch.from_numpy(pts).cuda()
    vals = torch.full((P,), float("nan"), dtype=torch.float64, device="cuda")
    plan.evaluate(cd, pd, vals)
    ref = O.evaluate_expansion(c, sup, pts)
    assert np.max(np.abs(vals.cpu().numpy() - ref)) <= 1e-12 * np.abs(c).sum()
    one = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    plan.evaluate(cd, pd[P - 1:], one)
    clone = plan.clone()
    again = torch.full((P,), float("nan"), dtype=torch.float64, device="cuda")
    clone.evaluate(cd, pd, again)
    torch.cuda.synchronize()
    assert one[0] == vals[P - 1] and torch.equal(again, vals)
    clone.close()
    plan.close()
