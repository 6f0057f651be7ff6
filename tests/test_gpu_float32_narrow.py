"""Float32 states with fewer than 32 trajectories: which step few long items take."""
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("B,degree,graphs", [(16, 230, 4), (8, 60, 20)])
def test_float32_below_32_trajectories(monkeypatch, B, degree, graphs):
    """few items: not the shared-memory kernel, however long the rows"""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2605_06921_gb300 as mq
    monkeypatch.setenv("MQO_TICK_KERNEL", "ticks")
    g = mi.erdos_renyi(500, degree / 500, 1)
    s = mq.Solver(mq.Graph(mi.pack([g] * graphs)), mq.params(problem=1, batch=B))
    assert s.info()["step_kernel"] == "staged"
