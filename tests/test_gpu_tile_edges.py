"""Kernels at the sizes where their tiles, chunks and splits end, against the FP64
oracles: absorbed BF16 rows of every residue of four columns, the FP64 apply with one
and with eight rows per warp, node-update chunks of each size, the warm-start network
at partial tiles, junction trees with long runs of equal intersections and long sums."""
import numpy as np
import pytest

import gen
from oracle import mlp as M
from oracle import tree_ot as O
from test_gpu_junction_general import compare_iterates, fp32_costs
from test_gpu_parity import marginal_gap, rel_err

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2406_10849_gb300 as T
    T.load()
    return T


@pytest.mark.parametrize("n,eps", [(5, 0.05), (130, 0.05), (255, 0.03), (516, 0.02), (1025, 0.02)])
def test_absorbed_rows_of_every_length(T, n, eps):
    """BF16 entries carry 2^-9 relative error: the phase's bounds as for the even sizes."""
    p = gen.prufer_problem(seed=7000 + n, J=6, n=n, num_leaves=3, eps=eps)
    with T.Solver([p], T.options(precision="fp32", apply_mode="bf16", lowp_start=2, absorb_tau=24)) as s:
        s.half_steps(8)
        got = s.potentials(0)
    ref = O.run_half_steps(p, 8)
    assert marginal_gap(p, got, ref) <= 3e-2
    assert rel_err(got, ref, p.eps) <= 5e-2


@pytest.mark.parametrize("count,n", [(1, 2), (1, 65), (3, 130), (640, 65)])
def test_fp64_rows_per_task(T, count, n):
    """640 chains hold more rows than one per warp of the GPU: the other split.  FP64 sums
    of n terms in another order: n 2^-53 relative, far below 1e-11."""
    probs = [gen.chain_problem(seed=7100 + i, J=3, n=n, eps=0.05) for i in range(count)]
    with T.Solver(probs, T.options(precision="fp64")) as s:
        s.half_steps(7)
        for i in {0, count // 2, count - 1}:
            assert rel_err(s.potentials(i), O.run_half_steps(probs[i], 7), probs[i].eps) <= 1e-11


def star(n, leaves, eps, seed):
    rng = np.random.default_rng(seed)
    fixed = np.ones(leaves + 1, bool)
    fixed[0] = False
    marg = {}
    for j in range(1, leaves + 1):
        m = rng.random(n) + 0.05
        marg[j] = m / m.sum()
    return gen.TreeProblem(name="star", edges=gen.star_edges(leaves), n=np.full(leaves + 1, n, np.int32), fixed=fixed,
                           marginals=marg, eps=eps, coords=[rng.random((n, 2)).astype(np.float32)] * (leaves + 1),
                           cost_scale=1.0)


@pytest.mark.parametrize("count,n,leaves", [(1, 1, 2), (1, 33, 8), (1, 257, 1), (2, 513, 5), (40, 641, 9), (260, 515, 10)])
def test_node_update_chunks(T, count, n, leaves):
    """From one pair to over 1.3 million (edge, point) pairs in a colour: each chunk size."""
    probs = [star(n, leaves, 0.1, 7200 + i) for i in range(count)]
    with T.Solver(probs, T.options(precision="fp32", autotune=False)) as s:
        s.half_steps(6)
        for i in {0, count - 1}:
            assert rel_err(s.potentials(i), O.run_half_steps(probs[i], 6), probs[i].eps) <= 1e-4


@pytest.mark.parametrize("dims,batch", [((1, 1, 1), 1), ((7, 33, 5), 31), ((64, 31, 65), 33), ((129, 96, 127), 1),
                                        ((40, 257, 32), 64)])
def test_network_at_partial_tiles(T, dims, batch):
    """The bounds of the full-size comparison: BF16 operands against a reference that rounds
    the same operands (2e-3 forward, 1e-2 gradients)."""
    i, h, o = dims
    rng = np.random.default_rng(7300 + batch)
    net = T.MLP(i, h, o, max_batch=64, seed=3)
    P = {k: v.astype(np.float64) for k, v in net.tensors(net.get_params()).items()}
    x = rng.normal(size=(batch, i)).astype(np.float32)
    t = rng.normal(size=(batch, o)).astype(np.float32)
    dev = torch.device("cuda")
    xd, td = torch.from_numpy(x).to(dev), torch.from_numpy(t).to(dev)
    y = torch.zeros(batch, o, device=dev)
    g = torch.zeros(net.num_params, device=dev)
    net.forward(xd, y)
    loss = net.backward(xd, td, g)
    torch.cuda.synchronize()

    def rel(a, b):
        return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-30))

    y_ref, _ = M.forward(P, x, bf16=True)
    loss_ref, g_ref = M.loss_and_grads(P, x, t, bf16=True)
    assert rel(y.cpu().numpy(), y_ref) <= 2e-3
    assert abs(loss - loss_ref) <= 2e-3 * loss_ref
    G = net.tensors(g.cpu().numpy())
    for name in ("W1", "b1", "W2", "b2", "W3", "b3"):
        assert rel(G[name], g_ref[name]) <= 1e-2, name


@pytest.mark.parametrize("J,d", [(1, 2), (9, 3), (12, 2), (2, 17)])
def test_junction_runs_and_long_sums(T, J, d):
    """Runs of 1 to 12 equal intersections; 17 points: sums over 17 and 289 entries per output."""
    jt = fp32_costs(gen.wls_junction_tree(7400 + J, J, d))
    for steps in (1, 4):
        compare_iterates(T, jt, steps)
