"""The multi-tick kernel of small member graphs against the tick's kernels:
the same machine (decisions, best sets, iterates, counters) and the same plain
steps, for every storage type, weights, ragged sizes and odd tick counts, and
with calls that alternate between the two."""
import numpy as np
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def mq():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2605_06921_gb300 as m
    return m


def graphs(weighted, B):
    gs = [mi.erdos_renyi(n, p, n) for n, p in ((33, 0.2), (1, 0.5), (90, 0.1), (64, 0.0))]
    if weighted:
        for g in gs:
            rows, cols = g.edges_directed()
            lo, hi = np.minimum(rows, cols), np.maximum(rows, cols)
            g.weights = np.where((lo * 7 + hi * 3) % 2, -1, 1).astype(np.int8)
    return mi.pack(gs)


@pytest.mark.parametrize("problem,weighted", [(0, False), (1, False), (1, True)])
@pytest.mark.parametrize("B,xd,vd", [(1, 0, 0), (2, 1, 1), (8, 0, 0), (16, 2, 0), (32, 1, 0), (128, 2, 2)])
def test_small_equals_ticks(mq, monkeypatch, problem, weighted, B, xd, vd):
    G = graphs(weighted, B)
    out = []
    for mode in ("small", "ticks"):
        monkeypatch.setenv("MQO_TICK_KERNEL", mode)
        s = mq.Solver(mq.Graph(G), mq.params(problem=problem, batch=B, x_dtype=xd, v_dtype=vd, t_gs=2,
                                             descent_cap=12, init_kind=1, sigma=0.2, seed=B,
                                             alpha=0.8 if problem == 0 else 0.05, momentum=0.4))
        assert s.info()["small"] == (mode == "small")
        s.run(1)
        s.run(178)
        s.step(3)
        stats = [t.cpu().tolist() for t in s.step_stats()]
        s.run(14)
        vals, bits = s.best()
        out.append((vals.tolist(), bits.cpu().tolist(), s.traj_state(), stats, s.get_x().float().cpu().tolist(),
                    s.get_v().float().cpu().tolist(), s.round().cpu().tolist()))
        s.reset()  # the other entry points see the state it left
        s.local_search()
        s.run(5)
        s.init()
        s.run(2)
        out[-1] += (s.traj_state(),)
    assert out[0] == out[1]


def test_small_default(mq):
    G = mi.erdos_renyi(200, 0.05, 0)
    assert mq.Solver(mq.Graph(G), mq.params(batch=1)).info()["small"]
    assert not mq.Solver(mq.Graph(G), mq.params(batch=1, pool_k=2)).info()["small"]
    assert not mq.Solver(mq.Graph(mi.erdos_renyi(3000, 0.01, 0)), mq.params(batch=32)).info()["small"]
