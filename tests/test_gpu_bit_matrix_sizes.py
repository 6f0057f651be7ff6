"""The kernels on bit matrices at the sizes their other tests leave out:
member graphs beyond 1024 nodes (a second word per lane) up to the largest
that has a matrix, CTAs that take several trajectory words or several pairs of
row tiles, and the autotuner where the multi-tick kernel is one of the plans."""
import numpy as np
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LARGEST = 1728  # nodes: 32 trajectories of x, masks and counters fill shared memory
DT = {1: torch.bfloat16, 2: torch.float16}


@pytest.fixture(scope="module")
def mq():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2605_06921_gb300 as m
    return m


def graph(sizes, p):
    made = {n: mi.erdos_renyi(n, p, n) for n in set(sizes)}
    return mi.pack([made[n] for n in sizes]) if len(sizes) > 1 else made[sizes[0]]


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("sizes,p,B", [
    ((1025,), 0.06, 32), ((1100, 300), 0.08, 64), ((LARGEST,), 0.06, 32),
    ((100,) * 160, 0.3, 64), ((100,) * 160, 0.3, 128), ((90,) * 60, 0.3, 128)])
def test_discrete_passes(mq, monkeypatch, problem, sizes, p, B):
    G = graph(sizes, p)
    g = mq.Graph(G)
    out = []
    monkeypatch.setenv("MQO_TICK_KERNEL", "ticks")
    for disc in ("bits", "pairs"):
        monkeypatch.setenv("MQO_DISC_KERNEL", disc)
        s = mq.Solver(g, mq.params(problem=problem, batch=B, x_dtype=1, t_gs=2, descent_cap=9, rho=0.5, init_kind=1,
                                   sigma=0.2, seed=B, momentum=0.4, alpha=0.8 if problem == 0 else 0.02))
        assert s.info()["disc_bits"] == (disc == "bits")
        s.run(120)
        a = s.traj_state()
        s.local_search()
        vals, bits = s.best()
        out.append((a, s.traj_state(), vals.tolist(), bits.cpu().tolist()))
    assert out[0] == out[1]


@pytest.mark.parametrize("sizes,p", [((1025, 40), 0.06), ((LARGEST,), 0.06)])
def test_evaluation(mq, sizes, p):
    G = graph(sizes, p)
    g = mq.Graph(G)
    B = 64
    rows, cols = G.edges_directed()
    off = np.asarray(G.node_offsets)
    gen = np.random.default_rng(3)
    for problem in (0, 1):
        s = mq.Solver(g, mq.params(problem=problem, batch=B, x_dtype=1))
        assert s.info()["disc_bits"]
        z = gen.random((G.n, B)) < (0.03 if problem == 0 else 0.5)
        got = [t.cpu().numpy() for t in s.evaluate(torch.from_numpy(mq.pack_bits(z, B)).cuda())]
        nb = np.zeros((G.n, B), dtype=np.int64)
        np.add.at(nb, rows, z[cols])
        deg = np.diff(G.row_ptr)[:, None]
        if problem == 0:
            node = (z, z * nb, ~z & (nb == 0))
        else:
            a = 2 * nb - deg
            node = (np.where(z, deg - nb, nb), ~np.where(z, a <= -1, a >= 0), np.where(z, a, -a) > 0)
        want = [np.add.reduceat(v.astype(np.int64), off[:-1], axis=0).reshape(-1) for v in node]
        want[problem == 0] //= 2  # both ends of a cut edge or a conflict
        for a, b in zip(got, want):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("sizes,p,B,xd", [
    ((1025,), 0.1, 32, 1), ((LARGEST,), 0.06, 32, 1), ((LARGEST, 900), 0.3, 64, 2), ((700,) * 120, 0.1, 128, 1)])
def test_dense_step(mq, monkeypatch, problem, sizes, p, B, xd):
    G = graph(sizes, p)
    g = mq.Graph(G)
    gen = torch.Generator(device="cuda").manual_seed(B + xd)
    lo = -problem
    x0 = ((torch.rand((G.n, B), device="cuda", generator=gen) - 0.45) * 2.4).clamp(lo, 1).to(DT[xd])
    out = []
    for force in ("dense", "generic"):
        monkeypatch.setenv("MQO_STEP_KERNEL", force)
        s = mq.Solver(g, mq.params(problem=problem, batch=B, x_dtype=xd, alpha=0.8 if problem == 0 else 0.02,
                                   momentum=0.4))
        assert s.info()["dense"] == (force == "dense")
        s.set_x(x0)
        s.step(4)
        out.append([s.get_x(), s.get_v(), *s.step_stats(), s.round()])
    for a, b in zip(*out):
        assert torch.equal(a, b)


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("B,xd", [(1, 0), (8, 1), (32, 1)])
def test_autotune_with_the_multi_tick_kernel(mq, monkeypatch, problem, B, xd):
    G = graph((60, 33, 90), 0.3)
    out = []
    for tune in (False, True):
        monkeypatch.setenv("MQO_TICK_KERNEL", "small" if tune and B == 8 else "ticks")
        s = mq.Solver(mq.Graph(G), mq.params(problem=problem, batch=B, x_dtype=xd, t_gs=2, descent_cap=9, rho=0.5,
                                             seed=B, momentum=0.4, alpha=0.8 if problem == 0 else 0.02))
        for ticks in (17, 40, 41):
            s.run(ticks)
            if tune:
                plan = s.autotune(5)
                assert plan["small"] == s.info()["small"]
        s.step(2)
        s.local_search()
        vals, bits = s.best()
        out.append((s.traj_state(), vals.tolist(), bits.cpu().tolist(), s.get_x().float().cpu().tolist()))
    assert out[0] == out[1]
