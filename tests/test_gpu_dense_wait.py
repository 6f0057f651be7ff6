"""A wait inside the tensor-core step kernel that runs out: every call on the
solver reports it once the kernel has marked it, the calls that synchronise
at once, and the context stays usable.  MQO_DENSE_POLLS=0: every wait has run
out before its first look."""
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CALLS = {
    "get_x": lambda s: s.get_x(),
    "get_v": lambda s: s.get_v(),
    "set_x": lambda s: s.set_x(torch.zeros((s.graph.n, s.B), dtype=torch.bfloat16, device="cuda")),
    "step_stats": lambda s: s.step_stats(),
    "round": lambda s: s.round(),
    "objective": lambda s: s.objective_f64(),
    "evaluate": lambda s: s.evaluate(s.bits_tensor()),
    "step": lambda s: s.step(1),
    "run": lambda s: s.run(1),
    "init": lambda s: s.init(),
    "reset": lambda s: s.reset(),
    "best": lambda s: s.best(),
    "traj_state": lambda s: s.traj_state(),
    "run_timed": lambda s: s.run_timed(1),
    "local_search": lambda s: s.local_search(),
    "autotune": lambda s: s.autotune(1),
}
SYNCHRONISE = ("best", "traj_state", "run_timed", "local_search", "autotune")


@pytest.fixture(scope="module")
def mq():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2605_06921_gb300 as m
    return m


def solver(mq, problem, sizes=(60, 300)):
    G = mi.pack([mi.erdos_renyi(n, 0.3, n) for n in sizes])
    s = mq.Solver(mq.Graph(G), mq.params(problem=problem, batch=32, x_dtype=1))
    assert s.info()["dense"]
    # points at the bounds: the rows go through the product
    x = (torch.arange(G.n * 32, device="cuda") % 3 == 0).view(G.n, 32).to(torch.bfloat16)
    s.set_x(x if problem == 0 else 2 * x - 1)
    return s


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("call,wait", [(c, True) for c in CALLS] + [(c, False) for c in SYNCHRONISE])
def test_every_call_reports_it(mq, monkeypatch, problem, call, wait):
    monkeypatch.setenv("MQO_STEP_KERNEL", "dense")
    monkeypatch.setenv("MQO_DENSE_POLLS", "0")
    s = solver(mq, problem)
    s.step(2)
    if wait:
        torch.cuda.synchronize()
    with pytest.raises(mq.MqoError) as e:
        CALLS[call](s)
    assert e.value.status == -5  # MQO_ETIMEOUT
    for c in CALLS:  # poisoned from here on
        with pytest.raises(mq.MqoError) as e:
            CALLS[c](s)
        assert e.value.status == -6, c  # MQO_ESTATE


def test_other_solvers_go_on(mq, monkeypatch):
    monkeypatch.setenv("MQO_STEP_KERNEL", "dense")
    monkeypatch.setenv("MQO_DENSE_POLLS", "0")
    bad = solver(mq, 0, (700, 130))
    monkeypatch.delenv("MQO_DENSE_POLLS")
    good, out = solver(mq, 0, (700, 130)), []
    for _ in range(3):
        try:
            bad.run(20)
        except mq.MqoError:
            pass
        good.step(1)
        out.append((good.get_x(), good.get_v(), *good.step_stats()))
    good.best()
    monkeypatch.setenv("MQO_STEP_KERNEL", "generic")
    ref = mq.Solver(good.graph, good.p)
    x = (torch.arange(830 * 32, device="cuda") % 3 == 0).view(830, 32).to(torch.bfloat16)
    ref.set_x(x)
    for got in out:
        ref.step(1)
        for a, b in zip(got, (ref.get_x(), ref.get_v(), *ref.step_stats())):
            assert torch.equal(a, b)
