"""Accuracy of the recomputed-cost messages on clustered supports, point by point: a few outliers
beside a dense cluster form groups far wider than the node's mean group."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import tree_ot as O


def message_errors(T, p, owner, nbr, **kw):
    """Errors, in nats, of the message to `owner` in the second half-step, against FP64 on the handle's own
    potentials, and the plan-weighted mean of C / eps per point."""
    with T.Solver([p], T.options(autotune=False, **kw)) as s:
        s.half_steps(1)
        f0 = s.potentials(0)
        s.half_steps(1)
        f1 = s.potentials(0)
        stats = s.plan_stats()
    C = O.cost(p, owner, nbr) / p.eps
    g = f0[(nbr, owner)] / p.eps
    a = g[None, :] - C
    top = a.max(1, keepdims=True)
    w = np.exp(a - top)
    m = top[:, 0] + np.log(w.sum(1))
    return f1[(owner, nbr)] / p.eps + m, (w * C).sum(1) / w.sum(1), stats


@pytest.mark.parametrize("dim", [1, 2, 3])
def test_outliers_beside_a_cluster(dim):
    """4096 points, 40 of them spread over the unit cube with 50 times the others' mass, the rest in a cluster of
    width 0.002.  The rms error over the outliers within the difference form's: a cost's FP32 rounding is at most
    (dim + 2) 2^-24 of it, its effect on the message the plan-weighted mean over the terms; 4 units of 2^-24 for
    the exponential, the operand and the sum."""
    import gen
    import paper_2406_10849_gb300 as T
    T.load()
    n, n_out = 4096, 40
    rng = np.random.default_rng(dim)
    centre = rng.random((1500, dim))
    x = 0.3 + 0.002 * rng.standard_normal((n, dim))
    x[n - n_out:] = rng.random((n_out, dim))
    mass = rng.random(n) + 0.5
    mass[n - n_out:] *= 50.0
    coords = [centre, x, rng.random((64, dim))]
    m2 = rng.dirichlet(np.ones(64))
    p = gen.TreeProblem(name="clustered", edges=gen.star_edges(2), n=np.array([1500, n, 64], np.int32),
                        fixed=np.array([False, True, True]), marginals={1: mass / mass.sum(), 2: m2 / m2.sum()},
                        eps=0.005, coords=[c.astype(np.float32) for c in coords], cost_scale=1.0)
    err, mean_cost, stats = message_errors(T, p, 1, 0)
    bound = ((dim + 2) * mean_cost + 4.0) * 2.0 ** -24
    out = slice(n - n_out, n)
    assert np.sqrt(np.mean(err[out] ** 2)) <= np.sqrt(np.mean(bound[out] ** 2))
    assert np.sqrt(np.mean(err ** 2)) <= np.sqrt(np.mean(bound ** 2))


def test_wide_groups_are_counted():
    """Uniform points have no wide group at these sizes; outliers beside a cluster have some, and few."""
    import gen
    import paper_2406_10849_gb300 as T
    T.load()
    rng = np.random.default_rng(5)
    flat = rng.random((4096, 2)).astype(np.float32)
    lumpy = (0.3 + 0.002 * rng.standard_normal((4096, 2))).astype(np.float32)
    lumpy[-40:] = rng.random((40, 2))
    m = {1: np.full(4096, 1.0 / 4096)}
    for x, lo, hi in ((flat, 0, 0), (lumpy, 40, 4096 // 8)):
        p = gen.TreeProblem(name="wide", edges=gen.star_edges(1), n=np.array([4096, 4096], np.int32),
                            fixed=np.array([False, True]), marginals=m, eps=0.01, coords=[flat, x], cost_scale=1.0)
        with T.Solver([p], T.options(autotune=False)) as s:
            st = s.plan_stats()
        assert st["factored_edges"] == 2
        assert lo <= st["wide_points"] <= hi


@pytest.mark.parametrize("k", [-24, 24])
@pytest.mark.parametrize("dim", [1, 2, 3])
def test_coordinates_in_other_units(dim, k):
    """Coordinates times 2^k, the cost scale divided by 2^(2 k): the same problem, every step of it scaled by a power
    of two, so the iterates agree bit for bit."""
    import gen
    import paper_2406_10849_gb300 as T
    T.load()
    rng = np.random.default_rng(dim)
    coords = [rng.random((n, dim)).astype(np.float32) for n in (700, 500, 900)]
    marg = {j: rng.dirichlet(np.ones(n)) for j, n in ((1, 500), (2, 900))}
    out = []
    for unit in (1.0, 2.0 ** k):
        p = gen.TreeProblem(name="units", edges=gen.star_edges(2), n=np.array([700, 500, 900], np.int32),
                            fixed=np.array([False, True, True]), marginals={j: m / m.sum() for j, m in marg.items()},
                            eps=0.1, coords=[c * np.float32(unit) for c in coords], cost_scale=unit ** -2.0)
        with T.Solver([p], T.options(autotune=False)) as s:
            assert s.plan_stats()["factored_edges"] == 4
            s.half_steps(4)
            out.append(s.potentials(0))
    for key in out[0]:
        assert np.array_equal(out[0][key], out[1][key]), key
