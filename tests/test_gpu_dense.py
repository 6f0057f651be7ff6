"""The tensor-core step kernel of dense member graphs against the plain
global-memory kernel: the same steps bit for bit, at the edges of its tiles,
for every storage type and relaxation, on the x its exact-sum argument does
not cover (small, out of the box, not a number) and at the bound of the one
it does."""
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


def both(mq, monkeypatch, G, x0, steps, **kw):
    """(dense, generic) outputs of `steps` plain steps from x0"""
    out = []
    for force in ("dense", "generic"):
        monkeypatch.setenv("MQO_STEP_KERNEL", force)
        s = mq.Solver(mq.Graph(G), mq.params(**kw))
        assert s.info()["dense"] == (force == "dense")
        s.set_x(x0)
        s.step(steps)
        out.append([s.get_x(), s.get_v(), *s.step_stats(), s.round()])
    return out


def same(a, b):
    for p, q in zip(a, b):
        if p.is_floating_point():
            ok = (p == q) | (torch.isnan(p) & torch.isnan(q))
            assert bool(ok.all())
        else:
            assert torch.equal(p, q)


def box(problem):
    return (0.0, 1.0) if problem == 0 else (-1.0, 1.0)


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("B,xd,vd", [(32, 1, 1), (64, 1, 0), (128, 2, 2), (32, 2, 0)])
@pytest.mark.parametrize("sizes", [(60,), (128, 17), (129, 255, 256, 257), (300, 641, 511)])
def test_dense_step_equals_generic(mq, monkeypatch, problem, B, xd, vd, sizes):
    gs = [mi.erdos_renyi(n, 0.3, n) for n in sizes]
    G = mi.pack(gs) if len(gs) > 1 else gs[0]
    lo, hi = box(problem)
    gen = torch.Generator(device="cuda").manual_seed(B + xd)
    for kind in ("clamped", "uniform"):
        r = torch.rand((G.n, B), device="cuda", generator=gen)
        x0 = r * (hi - lo) + lo if kind == "uniform" else ((r - 0.45) * 2.4).clamp(lo, hi)
        same(*both(mq, monkeypatch, G, x0.to(DT[xd]), 4, problem=problem, batch=B, x_dtype=xd, v_dtype=vd,
                   alpha=0.8 if problem == 0 else 0.02, momentum=0.4, gamma=1.7))


@pytest.mark.parametrize("objective", [1, 2, 3])
def test_dense_step_relaxations(mq, monkeypatch, objective):
    G = mi.pack([mi.erdos_renyi(n, 0.4, n) for n in (90, 140)])
    gen = torch.Generator(device="cuda").manual_seed(3)
    x0 = ((torch.rand((G.n, 32), device="cuda", generator=gen) - 0.5) * 3).clamp(-1, 1).to(torch.bfloat16)
    same(*both(mq, monkeypatch, G, x0, 5, problem=1, batch=32, x_dtype=1, alpha=0.02, momentum=0.4,
               objective=objective))


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("xd", [1, 2])
@pytest.mark.parametrize("spread", [1, 3, 99])
def test_dense_step_at_the_bound_of_exact_sums(mq, monkeypatch, problem, xd, spread):
    """odd significands down to the smallest x that counts as exact, degrees
    just below 2^8: every bit of the float32 sums is in use"""
    G = mi.pack([mi.erdos_renyi(250, 0.92, k) for k in range(2)])
    assert 200 < np.diff(G.row_ptr).max() < 256
    bits = 8 if xd == 1 else 11
    t = (17 if xd == 1 else 14) - 8
    gen = torch.Generator(device="cuda").manual_seed(5 + xd)
    e = torch.randint(0, min(spread, t), (G.n, 32), device="cuda", generator=gen).double()
    m = (torch.randint(2 ** (bits - 1), 2 ** bits, (G.n, 32), device="cuda", generator=gen) | 1).double()
    x0 = (m * 2.0 ** (1 - bits) * 2.0 ** (-1.0 - e)).to(DT[xd])
    if problem == 1:
        x0 = x0 * (torch.randint(0, 2, x0.shape, device="cuda", generator=gen) * 2 - 1).to(DT[xd])
    same(*both(mq, monkeypatch, G, x0, 1, problem=problem, batch=32, x_dtype=xd, v_dtype=0, alpha=1.0, momentum=0.4))


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("share", [0.0003, 0.02])
@pytest.mark.parametrize("value", [1e-6, 2.0 ** -11, float("nan"), float("inf"), -0.5, 3.0, -0.0])
def test_dense_step_irregular_x(mq, monkeypatch, problem, share, value):
    """a few (listed pairs) and many (rows summed again) doubtful x"""
    G = mi.pack([mi.erdos_renyi(150, 0.3, k) for k in range(3)])
    gen = torch.Generator(device="cuda").manual_seed(9)
    x0 = (torch.rand((G.n, 32), device="cuda", generator=gen) < 0.3).float()
    x0[torch.rand(x0.shape, device="cuda", generator=gen) < share] = value
    same(*both(mq, monkeypatch, G, x0.to(torch.bfloat16), 1, problem=problem, batch=32, x_dtype=1))


@pytest.mark.parametrize("problem", [0, 1])
def test_dense_machine_equals_generic(mq, monkeypatch, problem):
    """the whole machine: decisions, best sets and iterates"""
    G = mi.pack([mi.erdos_renyi(n, 0.25, n) for n in (140, 90, 128)])
    kw = dict(problem=problem, batch=32, x_dtype=1, t_gs=3, descent_cap=20, init_kind=1, sigma=0.1, seed=5,
              alpha=0.8 if problem == 0 else 0.01, momentum=0.4)
    out = []
    for force in ("dense", "generic"):
        monkeypatch.setenv("MQO_STEP_KERNEL", force)
        s = mq.Solver(mq.Graph(G), mq.params(**kw))
        assert s.info()["dense"] == (force == "dense")
        s.run(203)
        vals, bits = s.best()
        out.append((vals.tolist(), bits.cpu().tolist(), s.traj_state(), s.get_x().float().cpu().tolist()))
    assert out[0] == out[1]


def test_dense_step_default(mq):
    """the default for dense graphs; not for sparse, weighted, FP32 or narrow ones"""
    dense, sparse = mi.erdos_renyi(300, 0.2, 1), mi.erdos_renyi(600, 0.004, 1)
    assert mq.Solver(mq.Graph(dense), mq.params(batch=32, x_dtype=1)).info()["dense"]
    assert not mq.Solver(mq.Graph(sparse), mq.params(batch=32, x_dtype=1)).info()["dense"]
    assert not mq.Solver(mq.Graph(dense), mq.params(batch=32)).info()["dense"]
    assert not mq.Solver(mq.Graph(dense), mq.params(batch=16, x_dtype=1)).info()["dense"]
    rows, cols = dense.edges_directed()
    keep = rows < cols
    signed = mi.from_edges(dense.n, rows[keep], cols[keep], np.where(cols[keep] % 2, -1, 1))
    assert not mq.Solver(mq.Graph(signed), mq.params(problem=1, batch=32, x_dtype=1)).info()["dense"]
