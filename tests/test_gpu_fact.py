"""The factored recomputed-cost apply (compact groups of points) against the FP64
oracle, at the sizes where its groups, stages and chunks end: partial groups and
blocks, odd supports, one to many groups, a support beyond one sorted chunk, the
group sizes 64 / 32 / 16 and the difference form beside them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

from oracle import tree_ot as O
from test_gpu_parity import marginal_gap, rel_err


def cloud_star(n, dim, eps, seed, clustered=False, offset=0.0, scale=1.0):
    """A star with one leaf per entry of n[1:], random points; the first leaf has zeros in its marginal."""
    import gen
    rng = np.random.default_rng(seed)
    coords = []
    for k in n:
        x = rng.random((k, dim))
        if clustered:  # half of the points in one place, the rest spread: groups of very unequal extent
            x[: k // 2] = 0.25
        coords.append((offset + scale * x).astype(np.float32))
    J = len(n)
    fixed = np.ones(J, bool)
    fixed[0] = False
    marg = {}
    for j in range(1, J):
        m = rng.random(n[j]) + 0.05
        if j == 1 and n[j] > 3:
            m[:: 3] = 0.0
        marg[j] = m / m.sum()
    return gen.TreeProblem(name="cloud_star", edges=gen.star_edges(J - 1), n=np.array(n, np.int32), fixed=fixed,
                           marginals=marg, eps=eps, coords=coords, cost_scale=1.0 / (scale * scale))


CASES = {
    # (sizes, dim, eps): supports just below, at and above 32, 64, 128 points; odd and even
    "edges_1d": ((65, 31, 32, 33, 63, 64, 127, 129), 1, 0.2),
    "edges_2d": ((129, 31, 32, 33, 64, 65, 95, 191), 2, 0.2),
    "edges_3d": ((66, 32, 33, 67, 130, 257), 3, 0.5),
    "groups_mixed_2d": ((900, 300, 150, 700, 1100), 2, 0.01),   # 64, 32, 16 and the difference form
    "small_eps_2d": ((1500, 700, 400), 2, 0.002),
    "chunks_1d": ((4097, 70, 33), 1, 0.01),
    "many_points": ((70, 8200, 513), 2, 0.02),
    "clustered_2d": ((600, 333, 64), 2, 0.01),
    "shifted_scaled_2d": ((300, 257, 190), 2, 0.02),
}


@pytest.mark.parametrize("steps", [1, 2, 3, 8])
@pytest.mark.parametrize("name", sorted(CASES))
def test_iterates(name, steps):
    import paper_2406_10849_gb300 as T
    T.load()
    n, dim, eps = CASES[name]
    p = cloud_star(n, dim, eps, seed=11, clustered=name.startswith("clustered"),
                   offset=-37.5 if name.startswith("shifted") else 0.0, scale=5.0 if name.startswith("shifted") else 1.0)
    ref = O.run_half_steps(p, steps)
    for tune in (False, True):
        with T.Solver([p], T.options(autotune=tune)) as s:
            s.half_steps(steps)
            got = s.potentials(0)
        assert rel_err(got, ref, p.eps) <= 1e-4
        assert marginal_gap(p, got, ref) <= 1e-6  # the bar of every FP32 iterate


def test_first_step_far_frames():
    """Frames far from the messages (a warm start whose potentials jump by hundreds of eps): the groups whose
    sums leave the FP32 range are summed again by the difference form."""
    import paper_2406_10849_gb300 as T
    T.load()
    p = cloud_star((400, 300, 260), 2, 0.005, seed=3)
    rng = np.random.default_rng(0)
    f = {}
    for a, b in np.asarray(p.edges):
        for j, k in ((int(a), int(b)), (int(b), int(a))):
            f[(j, k)] = 2.0 * rng.random(int(p.n[j])) - 1.0  # up to 200 eps
    ref = O.run_half_steps(p, 2, f)
    with T.Solver([p], T.options()) as s:
        s.set_potentials(f)
        s.half_steps(2)
        got = s.potentials(0)
    assert rel_err(got, ref, p.eps) <= 1e-4
    assert marginal_gap(p, got, ref) <= 1e-6


def test_solve_certified_and_exact():
    import paper_2406_10849_gb300 as T
    T.load()
    p = cloud_star((500, 350, 420), 2, 0.01, seed=5)
    for kw in (dict(), dict(exact_dist=True)):
        with T.Solver([p], T.options(tol=1e-6, tol_kind="max", max_half_steps=20000, **kw)) as s:
            rc, res = s.solve()
            assert rc == 0
            fc = O.final_check(p, s.potentials(0))
        assert fc["max_marginal_l1"] <= 1e-6
