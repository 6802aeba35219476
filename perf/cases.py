"""The work that users of this library have it do, as cases to be timed.

A case is one call (or one prepared launch) through the package's public entry
points on a plan that the program keeps: the transform from samples to
Chebyshev coefficients (FP64 and mixed precision, both grid kinds, total-degree
and sparse supports, dimensions 2 to 100, alone and as a batch), and the way
back, the expansion's values at arbitrary points.  Supports, grids and
tolerances are those of this repository's workloads, tests and benchmark; the
target function of every state is drawn from its seed.
"""
import math

import numpy as np
import torch

import paper_2309_14584_gb300 as F
import workloads as W

OPTS = {
    "fp64": dict(precision=F.FCT_FP64, tol=1e-13),
    "mixed": dict(precision=F.FCT_MIXED, tol=1e-12, inner_tol=1e-4),
}


def _total(name, D, d, K, lo, hi, family, precision, grid_seed, first=False, block_threads=0):
    """One transform on the total-degree support |n|_1 <= d, K grids by Algorithm 1 with lo..hi points per axis."""
    return dict(name=name, kind="transform", support="total", D=D, d=d, N=math.comb(D + d, d), nonzeros=0, K=K, lo=lo,
                hi=hi, family=family, precision=precision, grid_seed=grid_seed, first=first,
                block_threads=block_threads)


def _sparse(name, D, d, N, nonzeros, K, precision, grid_seed, block_threads=0):
    """One transform on N multi-indices of max degree d with `nonzeros` nonzero components each."""
    return dict(name=name, kind="transform", support="sparse", D=D, d=d, N=N, nonzeros=nonzeros, K=K, lo=1, hi=d + 1,
                family="poly", precision=precision, grid_seed=grid_seed, first=False, block_threads=block_threads)


def listed():
    return [
        # the smallest transform users run (the smoke test's): 153 coefficients, latency only
        _total("d2_fp64", 2, 16, 4, 9, 33, "poly", "fp64", 1),
        # a mid-size analytic target in six dimensions, on either path
        _total("d6_fp64", 6, 10, 18, 1, 11, "gausscos", "fp64", 2),
        _total("d6_mixed", 6, 10, 18, 1, 11, "gausscos", "mixed", 2),
        # the benchmark's headline transform, on either path (512-thread blocks are the tuner's choice on the mixed one)
        _total("d10_mixed", 10, 8, 30, 1, 9, "rational", "mixed", 3, block_threads=512),
        _total("d10_fp64", 10, 8, 30, 1, 9, "rational", "fp64", 3),
        # a high-dimensional serving shape: many grids (Algorithm 2's choice), few degrees
        _total("d18_mixed", 18, 5, 171, 1, 6, "gausscos", "mixed", 5000033),
        # the paper's own first-kind grid (signed half entries, more iterations)
        _total("d6_first_kind", 6, 10, 18, 1, 11, "gausscos", "mixed", 2, first=True),
        # high degree in two dimensions: long axes, the DCT counts
        _total("d2_long_axis", 2, 300, 8, 150, 301, "gausscos", "mixed", 24),
        # sparse supports in a hundred dimensions: short indices on many grids, and longer ones at a larger N
        _sparse("sparse_d100", 100, 9, 20000, 3, 1000, "mixed", 300),
        _sparse("sparse10_d100", 100, 3, 50000, 10, 240, "mixed", 500, block_threads=512),
        # unlike transforms in one prepared launch (an engine's batch)
        dict(name="batch_mixed", kind="batch", B=48, dmin=3, dmax=8, degmin=6, degmax=10, per_dim=8,
             precision="mixed", grid_seed=4),
        # the way back: values of a six-dimensional expansion at many points
        dict(name="evaluate_d6", kind="evaluate", D=6, d=10, points=131072),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    seed = rng.randrange(1, 1 << 20)
    if u < 0.60:  # total-degree transforms, N from about a hundred to forty thousand
        D = rng.choice([2, 3, 4, 5, 6, 7, 8, 10, 12, 15, 20])
        n = _log_int(rng, 120, 40000)
        d = max(2, max(k for k in range(1, 400) if k == 1 or math.comb(D + k, k) <= n))
        if D == 2:
            K, lo, hi = rng.randint(4, 8), max(2, d // 2), 2 * d + 1
        else:
            K, lo, hi = rng.randint(6, 9) * D, 1, d + 1
        prec = rng.choice(["fp64", "mixed", "mixed"])
        first = D > 2 and d <= 10 and rng.random() < 0.1
        return {k: v for k, v in _total("", D, d, K, lo, hi, rng.choice(["gausscos", "rational", "poly"]), prec, seed,
                                        first, rng.choice([0, 0, 256, 512])).items() if k != "name"}
    if u < 0.75:  # sparse supports
        N = _log_int(rng, 2000, 20000)
        D = rng.choice([30, 60, 100])
        nz = rng.choice([3, 5, 10])
        K = rng.randint(500, 900) if nz == 3 else rng.randint(200, 300)
        return {k: v for k, v in _sparse("", D, 9 if nz == 3 else 3, N, nz, K, rng.choice(["fp64", "mixed", "mixed"]),
                                         seed, rng.choice([0, 512])).items() if k != "name"}
    if u < 0.88:
        return dict(kind="batch", B=rng.randint(3, 40), dmin=3, dmax=rng.randint(4, 8), degmin=6,
                    degmax=rng.randint(7, 10), per_dim=8, precision=rng.choice(["fp64", "mixed"]), grid_seed=seed)
    return dict(kind="evaluate", D=rng.choice([2, 3, 4, 6, 8]), d=rng.randint(3, 9), points=_log_int(rng, 1000, 120000))


# -- inputs -------------------------------------------------------------------
def _members(case):
    """(support, sizes, nodes) of every transform of the case."""
    if case["kind"] == "evaluate":
        D = case["D"]
        return [(W.total_degree_support(D, case["d"]),) + W.l_grid(1, 1, D, 1, 2, 3)]
    if case["kind"] == "batch":
        g = np.random.default_rng(case["grid_seed"])
        out = []
        for t in range(case["B"]):
            D, d = int(g.integers(case["dmin"], case["dmax"] + 1)), int(g.integers(case["degmin"], case["degmax"] + 1))
            sup = W.total_degree_support(D, d)
            out.append((sup,) + W.l_grid(case["grid_seed"] * 1_000_003 + t, len(sup), D, case["per_dim"] * D, 1, d + 1))
        return out
    D, d, N = case["D"], case["d"], case["N"]
    if case["support"] == "total":
        sup = W.total_degree_support(D, d)
    elif case["nonzeros"] == 3:
        sup = W.sparse_infinity_support(13, D, d, N, 3)
    else:
        sup = W.sparse_support_vectorised(3, D, d, N, case["nonzeros"])
    return [(sup,) + W.l_grid(case["grid_seed"], len(sup), D, case["K"], case["lo"], case["hi"])]


def _target(family, sup, seed):
    """(family code, parameters) of the seed's target function."""
    D = sup.shape[1]
    if family == "poly":
        return F.FCT_FAMILY_POLY, W.poly_coefficients(seed, sup)
    if family == "gausscos":
        return F.FCT_FAMILY_GAUSSCOS, W.gausscos_params(seed, D)
    return F.FCT_FAMILY_RATIONAL, W.rational_params(seed, D)


def _family(case):
    return "gausscos" if case["kind"] == "batch" else case["family"]


def _points(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return 2 * torch.rand(case["points"], case["D"], dtype=torch.float64, device="cuda", generator=g) - 1


def prepare(case, seed):
    members = _members(case)
    if case["kind"] == "evaluate":
        sup, sizes, nodes = members[0]
        plan = F.Plan(sup, sizes, nodes)
        c = torch.from_numpy(W.poly_coefficients(seed, sup)).cuda()
        return dict(kind="evaluate", plan=plan, c=c, points=_points(case, seed),
                    values=torch.empty(case["points"], dtype=torch.float64, device="cuda"))
    opts = dict(OPTS[case["precision"]], max_iter=20000)
    if case.get("first"):
        opts["grid_kind"] = F.FCT_GRID_FIRST_KIND
    if case.get("block_threads"):
        opts["block_threads"] = case["block_threads"]
    plans, xs, cs = [], [], []
    for t, (sup, sizes, nodes) in enumerate(members):
        p = F.Plan(sup, sizes, nodes, **opts)
        x = torch.empty(p.M, dtype=torch.float64, device="cuda")
        family, params = _target(_family(case), sup, seed * 4099 + t)
        p.sample(family | (F.fct.FCT_SAMPLE_FOLDED if family == F.FCT_FAMILY_POLY else 0), params, x)
        plans.append(p)
        xs.append(x)
        cs.append(torch.empty(p.N, dtype=torch.float64, device="cuda"))
    state = dict(kind=case["kind"], plans=plans, xs=xs, cs=cs)
    if case["kind"] == "batch":
        state["batch"] = _Batch([p.handle for p in plans], xs, cs)
    return state


class _Batch:
    """A prepared batch that is destroyed with its state."""

    def __init__(self, handles, xs, cs):
        self.handle = F.fct_batch_create(handles, xs, cs)

    def __del__(self):
        F.fct_batch_destroy(self.handle)


def run(state):
    if state["kind"] == "evaluate":
        state["plan"].evaluate(state["c"], state["points"], state["values"])
        return state["values"]
    if state["kind"] == "batch":
        F.fct_batch_launch(state["batch"].handle)
        return torch.cat(state["cs"])
    state["plans"][0].execute(state["xs"][0], state["cs"][0], report=False)
    return state["cs"][0]


# -- work ---------------------------------------------------------------------
def _iterations(case):
    """CG iterations the path takes, measured on these shapes (they vary by a few with the target)."""
    if case.get("first"):
        return 1240
    if case["kind"] == "batch":
        return 180
    if case["support"] == "sparse":
        return 260 if case["nonzeros"] == 3 else 700
    return {2: 20, 6: 150, 10: 440}.get(case["D"], 180) if case["K"] <= 3 * case["D"] or case["D"] == 2 else 250


def work(case):
    """Bytes: the samples in, the coefficients out, and per iteration the vectors s, p, x and q once (they fit the
    chip, the alias tables are implied by the plan).  Flops: the DCT passes by direct matrix products are not counted
    (a fast transform needs few), the two alias products of every iteration are (one multiply-add per entry each)."""
    if case["kind"] == "evaluate":
        n = math.comb(case["D"] + case["d"], case["d"])
        return {"bytes": 8.0 * (case["points"] * (case["D"] + 1) + n), "flops": 1.0 * case["points"] * n * case["D"]}
    total_b = total_f = 0.0
    w = 8.0 if case["precision"] == "fp64" else 4.0
    if case["kind"] == "batch":
        g = np.random.default_rng(case["grid_seed"])
        shapes = []
        for _ in range(case["B"]):
            D, d = int(g.integers(case["dmin"], case["dmax"] + 1)), int(g.integers(case["degmin"], case["degmax"] + 1))
            shapes.append((math.comb(D + d, d), case["per_dim"] * D))
    else:
        shapes = [(case["N"], case["K"])]
    for N, K in shapes:
        total_b += 8.0 * (1.5 * K * N + N) + _iterations(case) * w * 6 * N
        total_f += _iterations(case) * 4.0 * K * N
    return {"bytes": total_b, "flops": total_f}


# -- the same results in plain 64-bit torch -----------------------------------
def _node_positions(n, xi, first, dev):
    if n == 1:
        return torch.tensor([xi], dtype=torch.float64, device=dev)
    j = torch.arange(n, dtype=torch.float64, device=dev)
    return torch.cos(math.pi * (j + 0.5) / n) if first else torch.cos(math.pi * j / (n - 1))


def _dct_matrix(n, first, dev):
    k = torch.arange(n, dtype=torch.float64, device=dev)[:, None]
    j = torch.arange(n, dtype=torch.float64, device=dev)[None, :]
    if first:
        return torch.cos(math.pi * k * (2 * j + 1) / (2 * n)) / n
    e = torch.ones(n, dtype=torch.float64, device=dev)
    e[0] = e[-1] = 0.5
    return (2.0 / (n - 1)) * e[:, None] * e[None, :] * torch.cos(math.pi * ((k * j) % (2 * (n - 1))) / (n - 1))


def _least_squares(sup, sizes, nodes, family, params, first):
    """argmin |A c - b| from the definitions: samples on every grid, a DCT along every axis, the alias operator as
    index arrays, conjugate gradients on the normal equations until they make no more progress."""
    dev = "cuda"
    K, D = sizes.shape
    m = torch.from_numpy(sup.astype(np.int64)).to(dev)
    par = torch.from_numpy(np.asarray(params, dtype=np.float64)).to(dev)
    rows, vals, rhs, base = [], [], [], 0
    for l in range(K):
        act = [i for i in range(D) if sizes[l, i] >= 2]
        shape = [int(sizes[l, i]) for i in act] or [1]
        q = torch.zeros(shape, dtype=torch.float64, device=dev)
        lin = torch.zeros(shape, dtype=torch.float64, device=dev)
        idx = torch.zeros(m.shape[0], dtype=torch.int64, device=dev)
        val = torch.ones(m.shape[0], dtype=torch.float64, device=dev)
        for i in range(D):
            n = int(sizes[l, i])
            x = _node_positions(n, float(nodes[l, i]), first, dev)
            if i in act:
                view = [1] * len(shape)
                view[act.index(i)] = n
                x = x.reshape(view)
            q = q + par[i] * x * x
            if family == F.FCT_FAMILY_GAUSSCOS:
                lin = lin + par[D + i] * x
            mi = m[:, i]
            if n == 1:
                val = val * torch.cos(mi.double() * math.acos(float(nodes[l, i])))
            elif first:
                r, sgn = mi % (2 * n), 1.0 - 2.0 * ((mi // (2 * n)) % 2).double()
                half = (r == 0).double() + 0.5 * ((r > 0) & (r < n)).double() - 0.5 * (r > n).double()
                idx = idx * n + torch.where(r < n, r, torch.where(r > n, 2 * n - r, 0 * r))
                val = val * sgn * half
            else:
                r = mi % (2 * (n - 1))
                idx = idx * n + torch.minimum(r, 2 * (n - 1) - r)
        f = torch.exp(-q) * torch.cos(lin) if family == F.FCT_FAMILY_GAUSSCOS else 1.0 / (1.0 + q)
        for a, n in enumerate(shape):
            if n >= 2:
                f = torch.tensordot(_dct_matrix(n, first, dev), f, dims=([1], [a])).movedim(0, a)
        bins, inv = torch.unique(idx, return_inverse=True)
        rhs.append(f.reshape(-1)[bins])
        rows.append(inv + base)
        vals.append(val)
        base += bins.numel()
    rows, vals, b = torch.stack(rows), torch.stack(vals), torch.cat(rhs)
    flat = rows.reshape(-1)

    def a_mul(v):
        return torch.zeros(base, dtype=torch.float64, device=dev).index_add_(0, flat, (vals * v[None, :]).reshape(-1))

    def at_mul(r):
        return (vals * r[rows]).sum(0)

    c = torch.zeros(m.shape[0], dtype=torch.float64, device=dev)
    for _ in range(2):  # a second solve for what rounding left in the first
        s = at_mul(b - a_mul(c))
        p, gam = s.clone(), s.dot(s)
        g0 = gam if _ == 0 else g0
        d = torch.zeros_like(c)
        for it in range(6000):
            if it % 20 == 0 and float(gam) <= 1e-30 * float(g0):
                break
            ap = a_mul(p)
            alpha = gam / ap.dot(ap).clamp_min(1e-300)
            d = d + alpha * p
            s = s - alpha * at_mul(ap)
            new = s.dot(s)
            p = s + (new / gam.clamp_min(1e-300)) * p
            gam = new
        c = c + d
    return c


def exact(case, seed):
    members = _members(case)
    if case["kind"] == "evaluate":
        sup = torch.from_numpy(members[0][0].astype(np.int64)).cuda()
        c = torch.from_numpy(W.poly_coefficients(seed, members[0][0])).cuda()
        theta = torch.acos(_points(case, seed).clamp(-1, 1))
        out = []
        for t in theta.split(2048):
            term = c[None, :].expand(t.shape[0], -1)
            for i in range(case["D"]):
                tab = torch.cos(t[:, i, None] * torch.arange(case["d"] + 1, device="cuda")[None, :])
                term = term * tab[:, sup[:, i]]
            out.append(term.sum(1))
        return torch.cat(out)
    got = []
    for t, (sup, sizes, nodes) in enumerate(members):
        family, params = _target(_family(case), sup, seed * 4099 + t)
        if family == F.FCT_FAMILY_POLY:  # in the support's span: the least-squares solution is the polynomial itself
            got.append(torch.from_numpy(params).cuda())
        else:
            got.append(_least_squares(sup, sizes, nodes, family, params, bool(case.get("first"))))
    return torch.cat(got)
