"""Evaluation programs at the edges of their two builders (one block up to 16384
components, several beyond) and of the one block's tiles of 256 terms, on supports in
order and shuffled (the zero index anywhere): against the
oracle, bound 1e-12 sum |c|."""
import numpy as np
import pytest
import torch

import paper_2309_14584_gb300 as F
import workloads as W
from oracle import fct_oracle as O

pytestmark = pytest.mark.gpu

CASES = [(1, 3), (31, 4), (32, 4), (255, 4), (256, 4), (257, 4), (511, 5), (512, 5), (513, 5), (2047, 8), (2048, 8),
         (2049, 8)]


@pytest.mark.parametrize("shuffled", [False, True])
@pytest.mark.parametrize("N,D", CASES)
def test_matches_the_oracle(N, D, shuffled):
    sup = W.total_degree_support(D, 12 if D < 8 else 6)
    if shuffled:
        sup = sup[W.stream(8, "probe").permutation(len(sup))]
    sup = np.ascontiguousarray(sup[:N])
    assert len(sup) == N
    plan = F.Plan(sup, np.full((1, D), 1, dtype=np.int32))
    g = W.stream(94, "probe")
    c = g.standard_normal(N)
    pts = g.uniform(-1.0, 1.0, (37, D))
    vals = torch.full((37,), float("nan"), dtype=torch.float64, device="cuda")
    plan.evaluate(torch.from_numpy(c).cuda(), torch.from_numpy(pts).cuda(), vals)
    ref = O.evaluate_expansion(c, sup, pts)
    assert np.max(np.abs(vals.cpu().numpy() - ref)) <= 1e-12 * np.abs(c).sum()
    plan.close()
