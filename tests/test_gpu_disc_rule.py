"""When the discrete passes run on bit matrices by default: always while rounds
are rare; with short descents not where the neighbour lists were faster."""
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("problem,n,degree,graphs,B,t_gs,cap,bits", [
    (0, 100, 10, 152, 64, 60, 50, True), (0, 100, 10, 152, 64, 1, 6, False), (0, 200, 80, 152, 64, 1, 6, True),
    (1, 100, 30, 152, 64, 1, 6, True), (0, 100, 10, 152, 64, 60, 6, False), (1, 100, 30, 152, 64, 90, 6, True),
    (0, 800, 120, 1, 32, 60, 50, True), (0, 800, 120, 1, 32, 1, 6, False), (1, 800, 120, 8, 64, 1, 6, False),
    (0, 800, 120, 8, 64, 1, 6, True), (0, 300, 60, 8, 32, 1, 6, True)])
def test_default_form(monkeypatch, problem, n, degree, graphs, B, t_gs, cap, bits):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("half as many graphs as SMs are the line")
    import paper_2605_06921_gb300 as mq
    monkeypatch.setenv("MQO_TICK_KERNEL", "ticks")
    g = mi.erdos_renyi(n, degree / n, 1)
    G = mi.pack([g] * graphs) if graphs > 1 else g
    s = mq.Solver(mq.Graph(G), mq.params(problem=problem, batch=B, x_dtype=1, t_gs=t_gs, descent_cap=cap))
    assert s.info()["disc_bits"] == bits
