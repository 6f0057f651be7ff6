"""A shared-memory step of one wave does not share the SMs with the fused discrete
kernel while rounds are rare; the trajectories do not depend on the order."""
import numpy as np
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def solver(problem, n, degree, graphs, B, x_dtype, t_gs, cap):
    import paper_2605_06921_gb300 as mq
    bg = [mi.erdos_renyi(n, degree / n, k) for k in range(2)]
    g = mq.Graph(mi.pack([bg[k % 2] for k in range(graphs)]))
    return mq.Solver(g, mq.params(problem=problem, batch=B, x_dtype=x_dtype, t_gs=t_gs, descent_cap=cap, alpha=0.1,
                                  momentum=0.5, rho=0.6, sigma=0.1, init_kind=1, seed=7))


@pytest.mark.parametrize("problem,n,degree,graphs,B,x_dtype,t_gs,cap,first", [
    (1, 300, 60, 75, 64, 2, 90, 200, True), (1, 300, 60, 75, 128, 2, 90, 200, True),
    (1, 300, 60, 77, 64, 2, 90, 200, False),   # more items than SMs
    (1, 300, 60, 75, 64, 2, 1, 6, False),      # rounds follow one another
    (0, 200, 36, 76, 128, 1, 60, 50, True), (0, 200, 36, 38, 32, 1, 60, 50, False),
    (0, 120, 40, 100, 128, 0, 60, 50, True), (1, 500, 60, 76, 128, 1, 90, 200, False)])
def test_order(monkeypatch, problem, n, degree, graphs, B, x_dtype, t_gs, cap, first):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the number of SMs is the line")
    monkeypatch.setenv("MQO_TICK_KERNEL", "ticks")
    s = solver(problem, n, degree, graphs, B, x_dtype, t_gs, cap)
    assert s.info()["step_first"] == first
    s.init()
    s.run(cap + 40)
    vals, bits = s.best()
    monkeypatch.setenv("MQO_DISC_KERNEL", "pairs")
    r = solver(problem, n, degree, graphs, B, x_dtype, t_gs, cap)
    assert not r.info()["step_first"]
    r.init()
    r.run(cap + 40)
    want, wbits = r.best()
    np.testing.assert_array_equal(vals, want)
    assert torch.equal(bits, wbits)
