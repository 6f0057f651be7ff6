"""The discrete passes on bit matrices against the node-parallel list passes:
the same repair and local-search rounds, at tile and word edges, with one, many
and all trajectories of a word in a round, inside the machine and standalone,
and with the plan changed in mid-search."""
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


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("B,xd", [(32, 1), (64, 0), (128, 1)])
@pytest.mark.parametrize("sizes,p", [((40, 64, 33), 0.45), ((128, 129, 200), 0.2), ((600,), 0.08), ((40,) * 160, 0.3)])
def test_bits_equal_lists(mq, monkeypatch, problem, B, xd, sizes, p):
    gs = [mi.erdos_renyi(n, p, n) for n in sizes]
    G = mi.pack(gs) if len(gs) > 1 else gs[0]
    out = []
    monkeypatch.setenv("MQO_TICK_KERNEL", "ticks")
    for disc in ("bits", "pairs"):
        monkeypatch.setenv("MQO_DISC_KERNEL", disc)
        s = mq.Solver(mq.Graph(G), mq.params(problem=problem, batch=B, x_dtype=xd, t_gs=2, descent_cap=9, rho=0.5,
                                             init_kind=1, sigma=0.2, seed=B, momentum=0.4,
                                             alpha=0.8 if problem == 0 else 0.02))
        assert s.info()["discrete_kernel"] == ("graph" if disc == "bits" else "pairs")
        s.run(150)
        a = s.traj_state()
        s.local_search()
        if disc == "bits":
            s.autotune(3)  # tries the other forms from this state
        s.run(40)
        vals, bits = s.best()
        out.append((a, s.traj_state(), vals.tolist(), bits.cpu().tolist()))
    assert out[0] == out[1]
