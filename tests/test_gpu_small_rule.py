"""When mqo_run takes the multi-tick kernel, and that plain steps between ticks
take it all the same: results as with the tick's kernels throughout."""
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


@pytest.mark.parametrize("problem,n,degree,B,t_gs,cap,small", [
    (0, 200, 10, 1, 60, 50, True), (0, 200, 10, 1, 1, 6, True), (0, 100, 10, 8, 60, 50, True),
    (0, 100, 10, 64, 60, 50, False),  # bit-matrix rounds beside a step of a few us
    (1, 100, 10, 64, 60, 50, True),   # long descents without repairs
    (1, 100, 10, 64, 1, 6, False), (0, 100, 4, 64, 60, 50, True), (0, 100, 4, 64, 1, 6, False),
    (1, 400, 4, 16, 0, 2, False), (1, 100, 4, 16, 0, 2, True)])
def test_plan_of_ticks(mq, problem, n, degree, B, t_gs, cap, small):
    g = mq.Graph(mi.erdos_renyi(n, degree / n, 1))
    s = mq.Solver(g, mq.params(problem=problem, batch=B, x_dtype=1, t_gs=t_gs, descent_cap=cap))
    assert s.info()["small"] == small


@pytest.mark.parametrize("problem", [0, 1])
def test_steps_between_ticks(mq, monkeypatch, problem):
    g = mq.Graph(mi.pack([mi.erdos_renyi(n, 0.1, n) for n in (100, 57)]))
    out = []
    for kernel in (None, "ticks"):
        if kernel:
            monkeypatch.setenv("MQO_TICK_KERNEL", kernel)
        s = mq.Solver(g, mq.params(problem=problem, batch=64, x_dtype=1, t_gs=1, descent_cap=6, seed=2, momentum=0.4,
                                   alpha=0.8 if problem == 0 else 0.02))
        assert not s.info()["small"]
        for ticks, steps in ((33, 2), (1, 1), (20, 5)):
            s.run(ticks)
            s.step(steps)
            out.append([t.tolist() for t in s.step_stats()])
        vals, bits = s.best()
        out.append([s.traj_state(), vals.tolist(), bits.tolist(), s.get_x().tolist(), s.get_v().tolist()])
    assert out[:4] == out[4:]
