"""Exact evaluation and the double-precision objective of every batch size and
storage type, on graphs with and without bit matrices, against the dense
matrix product."""
import numpy as np
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("problem,weighted", [(0, False), (1, False), (1, True)])
@pytest.mark.parametrize("B,xd", [(1, 0), (4, 0), (8, 2), (16, 1), (32, 1), (64, 0), (128, 2)])
@pytest.mark.parametrize("p", [0.3, 0.02])
def test_readouts(problem, weighted, B, xd, p):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2605_06921_gb300 as mq
    G = mi.pack([mi.erdos_renyi(n, p, n) for n in (40, 257, 130)])
    rows, cols = G.edges_directed()
    if weighted:
        G.weights = np.where((rows + cols) % 3, 1, -1).astype(np.int8)
    A = np.zeros((G.n, G.n))
    A[rows, cols] = 1 if G.weights is None else G.weights
    s = mq.Solver(mq.Graph(G), mq.params(problem=problem, batch=B, x_dtype=xd, seed=3))
    z = (np.random.default_rng(B).random((G.n, B)) < 0.4).astype(np.int64)
    got = [t.cpu().numpy() for t in s.evaluate(torch.from_numpy(mq.pack_bits(z, B)).cuda())]
    x = s.get_x().double().cpu().numpy()
    obj = s.objective_f64().cpu().numpy()
    P, d = (A @ z).astype(np.int64), A.sum(1).astype(np.int64)[:, None]
    if problem == 0:
        node = [z, z * P, (z == 0) & (P == 0), x - x * (A @ x)]
    else:
        s2 = 2 * P - d
        node = [np.where(z, d - P, P), ~np.where(z, s2 <= -1, s2 >= 0), np.where(z, s2, -s2) > 0,
                -np.float64(np.float32(0.001)) * x - x * (A @ x)]
    sums = [np.add.reduceat(t.astype(np.float64), G.node_offsets[:-1], axis=0).reshape(-1) for t in node]
    sums[1 if problem == 0 else 0] /= 2  # every edge was counted from both ends
    for a, b in zip(got, sums):
        assert np.array_equal(a, b)
    # (Ax) in float32: at most 77 summands of at most 1, over 257 nodes
    assert np.abs(obj - sums[3]).max() <= 257 * 77 * 77 * 2.0 ** -24
