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
