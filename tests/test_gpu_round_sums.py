"""The sums behind the check and the rounding of FP32 handles: the largest cost among near-ties,
feasibility to FP64 rounding, and costs and masses near the ends of the FP32 range."""
import numpy as np
import pytest

import gen
from gen.problems import TreeProblem
from oracle import tree_ot as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2406_10849_gb300 as T
    T.load()
    return T


@pytest.mark.parametrize("dim,seed", [(2, 5), (2, 21), (2, 26), (3, 2), (3, 15), (3, 17), (3, 21)])
def test_largest_cost_among_near_ties(T, dim, seed):
    """Two opposite clusters a few FP32 units wide: 4096 costs that agree to FP32 rounding.  The largest one is that
    of double-float distances, exact to about 2^-45, whichever side holds the rows."""
    rng = np.random.default_rng(seed)
    at = np.array([0.61, 0.37, 0.29])[:dim]
    coords = [(sign * at * (1.0 + 1e-7 * rng.standard_normal((64, dim)))).astype(np.float32) for sign in (1.0, -1.0)]
    p = TreeProblem(name="ties", edges=np.array([[0, 1]], np.int32), n=np.array([64, 64], np.int32),
                    fixed=np.array([False, True]), marginals={1: np.full(64, 1.0 / 64)}, eps=0.2, coords=coords,
                    cost_scale=1.0, cost_kind="sqeuclid")
    want = O.c_infinity(p)
    with T.Solver([p], T.options(autotune=False)) as s:
        s.half_steps(2)
        for side in (0, 1):
            assert abs(s.round(side)[0]["c_inf"] - want) <= 2.0 ** -45 * want


def plans_of(s, p):
    return [s.round_plan(0, e).cpu().numpy() for e in range(p.num_edges)]


@pytest.mark.parametrize("n", [2, 20, 63, 200])
@pytest.mark.parametrize("kind", ["sqeuclid", "dense"])
@pytest.mark.parametrize("steps", [1, 6])
def test_feasible_to_fp64_rounding(T, n, kind, steps):
    """Fixed marginals of the rounded plans in L1, in units of 2^-53: one rounding each for the target, the scales x
    and y, err_r, err_c, E and the entry's products, and the sums of this test (pairwise) beside them: 8; and one
    for every FP64 addition of a task of 64 rows to a column's sum, in an order that changes from run to run."""
    rng = np.random.default_rng(n)
    p = gen.random_tree_problem(rng, 4, n_range=(n, n + 13), eps_range=(0.05, 0.05), D=2, name="gap")
    p.cost_kind = kind
    with T.Solver([p], T.options(autotune=False)) as s:
        s.half_steps(steps)
        s.round()
        plans = plans_of(s, p)
    worst = 0.0
    for plan, (a, b) in zip(plans, np.asarray(p.edges)):
        for j, q in ((int(a), plan.sum(1)), (int(b), plan.sum(0))):
            if p.fixed[j]:
                worst = max(worst, float(np.abs(q - p.marginals[j] / p.marginals[j].sum()).sum()))
    assert worst <= (8.0 + (n + 13 + 63) // 64) * 2.0 ** -53


@pytest.mark.parametrize("k", [-90, 90])
def test_costs_in_other_units(T, k):
    """Stored costs and eps times 2^k: the same entries, so every cost of the rounding scales by 2^k but for the
    order of its FP64 additions."""
    p = gen.chain_problem(seed=1001, n=70, eps=0.05)
    costs = [p.dense_cost(e).astype(np.float32) for e in range(p.num_edges)]
    out = []
    for unit in (1.0, 2.0 ** k):
        q = gen.chain_problem(seed=1001, n=70, eps=0.05)
        q.eps = p.eps * unit
        dev = [torch.tensor(c * np.float32(unit), device="cuda") for c in costs]
        with T.Solver([q], T.options(autotune=False), device_costs=[dev]) as s:
            s.half_steps(5)
            r = s.round()[0]
            out.append([r[key] / unit for key in ("transport_cost", "rounded_transport_cost", "c_inf")])
    for a, b in zip(*out):
        assert abs(a - b) <= 1e-13 * abs(a)


def test_masses_beyond_the_fp32_range(T):
    """Potentials 89.5 eps too large: entries fit FP32, the sums over a row of three do not.  Check and rounding
    report what FP64 sums of the same entries give."""
    n = 3
    m = np.array([0.05, 0.9, 0.05])
    coords = [np.linspace(0.0, 0.1, n)[:, None].astype(np.float32) for _ in range(2)]
    p = TreeProblem(name="heavy", edges=np.array([[0, 1]], np.int32), n=np.array([n, n], np.int32),
                    fixed=np.array([False, True]), marginals={1: m}, eps=1.0, coords=coords, cost_scale=1.0,
                    cost_kind="sqeuclid")
    C = O.cost(p, 0, 1)
    f01 = np.log(np.full(n, 1.0 / n)) + 89.5
    f = {(0, 1): f01, (1, 0): np.zeros(n)}
    B = np.exp(f01[:, None] + np.log(m)[None, :] - C)
    assert B.max() < 3.4e38 and B.sum() > 3.4e38 and B.sum(0).max() > 3.4e38
    with T.Solver([p], T.options(autotune=False)) as s:
        s.half_steps(2)
        s.set_potentials(f)
        chk = s.check()[0]
        for side in (0, 1):
            r = s.round(side)[0]
            assert r["transport_cost"] == pytest.approx(float((B * C).sum()), rel=1e-6)
            plan = s.round_plan(0, 0).cpu().numpy()
            assert np.abs(plan.sum(0) - m).sum() <= 1e-13 and abs(plan.sum() - 1.0) <= 1e-13
    assert chk["transport_cost"] == pytest.approx(float((B * C).sum()), rel=1e-6)
