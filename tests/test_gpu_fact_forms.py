"""Every form of the factored recomputed-cost apply, fixed by a test option instead of the
autotuner's timing: one warp per block of outputs or 2, 4, 8 warps sharing it, in a launch of its
own or in one with the difference form, and its fallback for frames that moved far.  Group sizes
64, 32 and 16, 1 to 3 dimensions, neighbours with fewer stages of 64 points than warps sharing them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import tree_ot as O
from test_gpu_fact import cloud_star
from test_gpu_parity import marginal_gap, rel_err

FORMS = [(split, both) for both in (0, 1) for split in range(4)]
SHAPES = {
    # (sizes, dim, eps)
    "few_stages_1d": ((65, 32, 33, 63, 64, 129), 1, 0.2),
    "few_stages_3d": ((66, 32, 33, 64, 130), 3, 0.5),
    "sizes_64_32_16_and_difference_2d": ((900, 300, 150, 700, 1100), 2, 0.01),
    "chunks_1d": ((4097, 70, 33), 1, 0.01),
    "many_points_2d": ((70, 4133, 513), 2, 0.02),
}


def solver(T, p, split, both, **kw):
    s = T.Solver([p], T.options(test_apply=(split, both), **kw))
    st = s.plan_stats()
    assert st["factored_split"] == split and st["both_forms"] == both
    return s


@pytest.mark.parametrize("exact", [False, True])
@pytest.mark.parametrize("split,both", FORMS)
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_iterates(name, split, both, exact):
    import paper_2406_10849_gb300 as T
    T.load()
    n, dim, eps = SHAPES[name]
    p = cloud_star(n, dim, eps, seed=21)
    with solver(T, p, split, both, exact_dist=exact) as s:
        if not exact:
            assert s.plan_stats()["factored_edges"] > 0
        for steps in (2, 3):
            s.reset()
            s.half_steps(steps)
            got = s.potentials(0)
            ref = O.run_half_steps(p, steps)
            assert rel_err(got, ref, p.eps) <= 1e-4
            assert marginal_gap(p, got, ref) <= 1e-6  # the bar of every FP32 iterate


@pytest.mark.parametrize("split,both", FORMS)
@pytest.mark.parametrize("n,dim,eps", [((400, 300, 260), 1, 0.002), ((1300, 33, 64, 2200), 2, 0.005),
                                       ((700, 900, 40), 3, 0.05)])
def test_fallback_of_far_frames(n, dim, eps, split, both):
    """Potentials that jump by hundreds of eps from point to point: frames far from the messages, sums out of
    the FP32 range.  Those groups are summed by the difference form, and the count shows that it ran.

    Bound on a message, in nats: a cost formed in FP32 has a relative error of (dim + 2) 2^-24, and with such
    potentials the largest costs count; 64 units of 2^-24 for the argument's, the exponential's and the sum's
    roundings.  Two half-steps, and a node's mean over its edges: three times that."""
    import paper_2406_10849_gb300 as T
    T.load()
    p = cloud_star(n, dim, eps, seed=3)
    rng = np.random.default_rng(0)
    f = {}
    for a, b in np.asarray(p.edges):
        for j, k in ((int(a), int(b)), (int(b), int(a))):
            f[(j, k)] = 200.0 * eps * (2.0 * rng.random(int(p.n[j])) - 1.0)
    ref = O.run_half_steps(p, 2, f)
    with solver(T, p, split, both) as s:
        assert s.plan_stats()["factored_edges"] > 0
        s.set_potentials(f)
        before = s.plan_stats()["factored_fallbacks"]
        s.half_steps(2)
        assert s.plan_stats()["factored_fallbacks"] > before
        got = s.potentials(0)
    worst = max(float(O.cost(p, int(a), int(b)).max()) for a, b in np.asarray(p.edges))
    bound = ((dim + 2) * worst / eps + 64.0) * 2.0 ** -24
    assert max(float(np.abs(got[k] - ref[k]).max()) for k in ref) / eps <= 3.0 * bound


@pytest.mark.parametrize("split", range(4))
@pytest.mark.parametrize("n,dim", [(8200, 1), (6001, 2), (4096, 3)])
def test_fallback_sums_long_supports(n, dim, split):
    """A message shifted by hundreds of binades since the last half-step: every group's sum over a long support
    comes from the fallback.  rms error in nats: a cost's FP32 rounding, (dim + 2) 2^-24 of it, weighted by the
    terms, and 4 units of 2^-24 for the exponential, the operand and the sum."""
    import gen
    import paper_2406_10849_gb300 as T
    T.load()
    rng = np.random.default_rng(dim)
    coords = [rng.random((k, dim)).astype(np.float32) for k in (n, 300, 64)]
    marg = {1: rng.dirichlet(np.ones(300)), 2: rng.dirichlet(np.ones(64))}
    p = gen.TreeProblem(name="long", edges=gen.star_edges(2), n=np.array([n, 300, 64], np.int32),
                        fixed=np.array([False, True, True]), marginals={k: m / m.sum() for k, m in marg.items()},
                        eps=0.5, coords=coords, cost_scale=1.0)
    with solver(T, p, split, 0) as s:
        s.half_steps(3)
        f = s.potentials(0)
        f[(0, 1)] = f[(0, 1)] + 150.0 * p.eps
        s.set_potentials(f)
        f = s.potentials(0)
        before = s.plan_stats()["factored_fallbacks"]
        s.half_steps(1)
        assert s.plan_stats()["factored_fallbacks"] - before >= 300 // 64
        got = s.potentials(0)[(1, 0)] / p.eps
    C = O.cost(p, 1, 0) / p.eps
    a = f[(0, 1)][None, :] / p.eps - C
    top = a.max(1, keepdims=True)
    w = np.exp(a - top)
    err = got + top[:, 0] + np.log(w.sum(1))
    bound = ((dim + 2) * (w * C).sum(1) / w.sum(1) + 4.0) * 2.0 ** -24
    assert np.sqrt(np.mean(err ** 2)) <= np.sqrt(np.mean(bound ** 2))


@pytest.mark.parametrize("tune", [False, True])
@pytest.mark.parametrize("n,dim,eps,splits", [
    ((64, 16384, 33), 2, 0.05, True), ((16385, 64, 65), 1, 0.05, True), ((130, 9001), 3, 0.5, True),
    ((70, 8255, 40), 2, 0.05, True), ((1024, 1024, 1024), 2, 0.01, False)])
def test_long_reductions_are_split(n, dim, eps, splits, tune):
    """Edges between a short and a long support: the long reduction is shared by the eight warps of a CTA and
    split over CTAs, where an even one keeps a single piece; splits that end in a partial stage or an odd point."""
    import paper_2406_10849_gb300 as T
    T.load()
    p = cloud_star(n, dim, eps, seed=8)
    with T.Solver([p], T.options(autotune=tune)) as s:
        st = s.plan_stats()
        assert st["factored_edges"] > 0
        assert (st["factored_splits"] > 1) == splits
        if splits and not tune:
            assert st["factored_split"] == 3
        for steps in (2, 3):
            s.reset()
            s.half_steps(steps)
            got = s.potentials(0)
            ref = O.run_half_steps(p, steps)
            assert rel_err(got, ref, p.eps) <= 1e-4
            assert marginal_gap(p, got, ref) <= 1e-6  # the bar of every FP32 iterate


def test_exact_distances_take_the_difference_form():
    """With exact squared distances from the start nothing is factored, and the reduction is cut into pieces of
    512 points as for every difference-form apply: 4 blocks of 1024 outputs x 8 pieces for each of the two leaves."""
    import paper_2406_10849_gb300 as T
    T.load()
    p = cloud_star((4096, 4096, 4000), 2, 0.05, seed=4)
    with T.Solver([p], T.options(exact_dist=True, autotune=False)) as s:
        st = s.plan_stats()
        assert st["factored_edges"] == 0
        assert st["apply_tasks_c0"] == 2 * 4 * 8 and st["apply_tasks_c1"] == 2 * 4 * 8


@pytest.mark.parametrize("persistent", [False, True])
def test_certification_switches_to_the_exact_plan_and_back(persistent):
    """16 x 16 stars certified at 1.2e-7: where the plain costs stop short of it, the handle goes on with exact
    distances, the difference form and its own splits; a reset brings the factored form back, bit for bit."""
    import gen
    import paper_2406_10849_gb300 as T
    T.load()
    probs = gen.warmstart_stars(9_000_000, 16, side=16, eps=0.005)
    with T.Solver(probs, T.options(tol=1.2e-7, tol_kind="max", max_half_steps=6000, autotune=False,
                                   persistent=persistent)) as s:
        assert s.plan_stats()["factored_edges"] > 0
        s.half_steps(6)
        first = [s.potentials(i) for i in (0, 9)]
        s.reset()
        rc, res = s.solve()
        assert s.plan_stats()["exact_plan"] == 1
        assert rc == 0
        for i in (0, 9):
            assert O.final_check(probs[i], s.potentials(i))["max_marginal_l1"] <= 1.5e-7
        s.reset()
        assert s.plan_stats()["exact_plan"] == 0
        s.half_steps(6)
        for i, f in zip((0, 9), first):
            again = s.potentials(i)
            assert all(np.array_equal(f[k], again[k]) for k in again)


def test_new_points_of_known_sizes_are_not_timed_again():
    """The autotuner's choice is kept per sizes and forms: another batch of points and eps on the same trees, which
    groups its points differently, takes it over."""
    import gen
    import paper_2406_10849_gb300 as T
    T.load()
    timed = []
    for seed in range(4):
        rng = np.random.default_rng(seed)
        probs = []
        for n in ((333, 301, 77), (205, 411, 1033, 90)):
            p = cloud_star(n, 2, float(np.exp(rng.uniform(np.log(0.01), np.log(0.03)))), seed=seed)
            probs.append(p)
        with T.Solver(probs, T.options()) as s:
            st = s.plan_stats()
        assert 0 < st["factored_edges"] < st["directed_edges"]
        timed.append(st["timed_configs"])
    assert timed[0] > 0 and timed[1:] == [0, 0, 0]


@pytest.mark.parametrize("split", range(4))
@pytest.mark.parametrize("n,dim,eps,clustered,sizes", [
    ((900, 700, 450, 1300, 260), 1, 0.002, False, (64, 32, 16)),
    ((577, 1215, 1480, 802, 940, 1895), 2, 0.01, False, (64, 32, 16)),
    ((900, 700, 450, 1300), 3, 0.05, False, (64, 32)), ((1470, 40), 3, 0.05, True, (16,))])
def test_group_sizes(n, dim, eps, clustered, sizes, split):
    """Nodes of every group size in every dimension, each with one and several warps per block."""
    import paper_2406_10849_gb300 as T
    T.load()
    p = cloud_star(n, dim, eps, seed=21, clustered=clustered)
    with solver(T, p, split, 0) as s:
        st = s.plan_stats()
        for gs in sizes:
            assert st[f"nodes_in_{gs}"] > 0, gs
        for steps in (2, 3):
            s.reset()
            s.half_steps(steps)
            got = s.potentials(0)
            ref = O.run_half_steps(p, steps)
            assert rel_err(got, ref, p.eps) <= 1e-4
            assert marginal_gap(p, got, ref) <= 1e-6  # the bar of every FP32 iterate


@pytest.mark.parametrize("split", range(4))
def test_persistent_launch_of_split_reductions(split):
    """The persistent launch runs the same tasks, with several reduction splits per edge, wide groups and both forms:
    the same bits as per-half-step launches."""
    import paper_2406_10849_gb300 as T
    T.load()
    probs = [cloud_star((64, 16384, 33), 2, 0.05, seed=1), cloud_star((300, 257, 45), 2, 0.003, seed=2),
             cloud_star((600, 333, 64), 2, 0.01, seed=3, clustered=True)]
    out = []
    for persistent in (False, True):
        with T.Solver(probs, T.options(autotune=False, persistent=persistent, test_apply=(split, 0))) as s:
            st = s.plan_stats()
            assert st["factored_splits"] > 1 and st["persistent"] == (2 if persistent else 0)
            assert 0 < st["factored_edges"] < st["directed_edges"]
            s.half_steps(5)
            out.append([s.potentials(i) for i in range(3)])
    for a, b in zip(*out):
        for k in a:
            assert np.array_equal(a[k], b[k]), k
