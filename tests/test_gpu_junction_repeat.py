"""The junction tree's stopping quantity and transport cost are the same bits on every call: their sums
over more than one CTA have a fixed order."""
import numpy as np
import pytest

import gen

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("J,d", [(3, 12), (4, 20), (6, 40)])
def test_sums_repeat(J, d):
    import paper_2406_10849_gb300 as T
    from paper_2406_10849_gb300.treeot import JunctionSolver
    T.load()
    jt = gen.wls_junction_tree(11, J, d)
    jt.clique_costs = [np.asarray(c, np.float32).astype(np.float64) for c in jt.clique_costs]
    jt.eps = 0.05
    with JunctionSolver(jt) as s:
        s.half_steps(3)
        first = (s.residual(), s.transport_cost())
        for _ in range(200):
            assert (s.residual(), s.transport_cost()) == first
