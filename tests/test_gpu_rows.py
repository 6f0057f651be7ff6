"""The row-group step kernel against the plain global-memory
kernel: the same steps, statistics and bits, at degrees around its batches of
four neighbours, slices longer than its staged column indices, packed graphs,
signed weights, and x out of the box or not a number."""
import numpy as np
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DT = {1: torch.bfloat16, 2: torch.float16}


@pytest.fixture(scope="module")
def mq():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2605_06921_gb300 as m
    return m


def signed(G):
    u, v = G.edges_directed()
    keep = u < v
    return mi.from_edges(G.n, u[keep], v[keep], np.where((u[keep] * 7 + v[keep]) % 3 == 0, -1, 1))


def graph(name):
    return {
        "regular": lambda: mi.random_regular(4002, 3, 1),
        "ragged": lambda: mi.erdos_renyi(1500, 0.003, 2),         # isolated nodes, degrees 0 to about 14
        "long_rows": lambda: mi.erdos_renyi(600, 0.36, 3),        # degrees of about 216 (at most 255)
        "packed": lambda: mi.pack([mi.erdos_renyi(n, 0.02, n) for n in (1, 7, 255, 256, 257, 900)]),
        "signed": lambda: signed(mi.erdos_renyi(2000, 0.004, 5)),
        "signed_packed": lambda: mi.pack([signed(mi.erdos_renyi(n, 0.03, n)) for n in (20, 300, 512)]),
    }[name]()


def both(mq, monkeypatch, G, x0, steps, **kw):
    out = []
    for force in ("rows", "generic"):
        monkeypatch.setenv("MQO_STEP_KERNEL", force)
        s = mq.Solver(mq.Graph(G), mq.params(alpha=0.05, momentum=0.6, lambda_=0.3, gamma=1.7, **kw))
        assert s.info()["step_kernel"] == ("rows" if force == "rows" else "global")
        s.set_x(x0)
        s.step(steps)
        out.append([s.get_x(), s.get_v(), *s.step_stats(), s.round()])
    for p, q in zip(*out):
        if p.is_floating_point():
            assert bool(((p == q) | (torch.isnan(p) & torch.isnan(q))).all())
        else:
            assert torch.equal(p, q)


@pytest.mark.parametrize("B,xd,vd", [(32, 1, 1), (64, 1, 0), (128, 2, 2), (64, 2, 0), (128, 1, 0)])
@pytest.mark.parametrize("problem,name", [(1, n) for n in ("regular", "ragged", "long_rows", "packed", "signed",
                                                           "signed_packed")]
                         + [(0, n) for n in ("regular", "ragged", "long_rows", "packed")])
def test_rows_step_equals_generic(mq, monkeypatch, problem, name, B, xd, vd):
    G = graph(name)
    gen = torch.Generator(device="cuda").manual_seed(B + xd)
    x0 = ((torch.rand((G.n, B), device="cuda", generator=gen) - 0.5) * 2.6).clamp(-problem, 1)
    both(mq, monkeypatch, G, x0.to(DT[xd]), 4, problem=problem, batch=B, x_dtype=xd, v_dtype=vd)


@pytest.mark.parametrize("problem,name", [(1, "ragged"), (1, "signed"), (0, "ragged")])
@pytest.mark.parametrize("value", [1e-6, float("nan"), float("inf"), 3.0, -0.0])
def test_rows_step_irregular_x(mq, monkeypatch, problem, name, value):
    G = graph(name)
    gen = torch.Generator(device="cuda").manual_seed(9)
    x0 = torch.rand((G.n, 32), device="cuda", generator=gen) * 2 - 1
    x0[torch.rand(x0.shape, device="cuda", generator=gen) < 0.02] = value
    both(mq, monkeypatch, G, x0.to(torch.bfloat16), 1, problem=problem, batch=32, x_dtype=1)


@pytest.mark.parametrize("problem,name", [(0, "packed"), (1, "packed"), (1, "signed")])
def test_rows_machine_equals_generic(mq, monkeypatch, problem, name):
    """the whole machine: trajectories that do not step keep x and V"""
    G = graph(name)
    out = []
    for force in ("rows", "generic"):
        monkeypatch.setenv("MQO_STEP_KERNEL", force)
        s = mq.Solver(mq.Graph(G), mq.params(problem=problem, batch=32, x_dtype=1, alpha=0.1, momentum=0.5, t_gs=3,
                                             descent_cap=20, init_kind=1, sigma=0.1, seed=5))
        s.run(203)
        vals, bits = s.best()
        out.append((vals.tolist(), bits.cpu().tolist(), s.traj_state(), s.get_x().float().cpu().tolist()))
    assert out[0] == out[1]


def test_rows_step_default(mq, monkeypatch):
    """the default with 16-bit x outside shared memory, in shared memory for few member graphs; not for the other
    relaxations, FP32 x, narrow batches, or a longest row that the rest of the step does not cover"""
    for name in ("MQO_STEP_KERNEL", "MQO_STEP_ELL", "MQO_COL16"):
        monkeypatch.delenv(name, raising=False)
    G = mq.Graph(mi.random_regular(40000, 3, 1))
    kern = lambda g, **kw: mq.Solver(g, mq.params(**{**dict(problem=1, batch=64, x_dtype=1), **kw})).info()["step_kernel"]
    assert kern(G) == kern(G, problem=0) == kern(G, x_dtype=2, v_dtype=0) == "rows"
    for kw in (dict(objective=1), dict(x_dtype=0), dict(batch=16)):
        assert kern(G, **kw) != "rows"
    hub = mi.from_edges(4002, np.zeros(256, dtype=np.int64), np.arange(1, 257))
    assert kern(mq.Graph(hub)) != "rows" and kern(mq.Graph(hub), problem=0) == "staged"
    assert kern(mq.Graph(mi.erdos_renyi(300, 0.02, 1)), problem=0) == "staged"     # fits in shared memory, two items
    many = mi.pack([mi.erdos_renyi(100, 0.2, 1)] * 200)
    assert kern(mq.Graph(many)).startswith("smem")
