"""Where the tensor-core step is the default: row tiles times trajectory groups
that fill the GPU, and the measured lines of the mean degree on both sides."""
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("problem,n,degree,graphs,B,dense", [
    (0, 1000, 100, 8, 128, True), (1, 1000, 100, 8, 128, True),    # 256 tiles
    (0, 1000, 100, 1, 32, False), (0, 1000, 100, 1, 128, False),   # 8 and 32
    (0, 1000, 200, 1, 128, True), (0, 850, 110, 4, 32, False),
    (1, 1000, 200, 1, 32, False), (1, 800, 110, 1, 128, False), (1, 800, 160, 1, 128, True),
    (1, 150, 80, 64, 32, False), (1, 150, 80, 64, 64, True), (1, 600, 100, 64, 32, True),
    (0, 600, 64, 16, 32, False), (0, 600, 100, 16, 32, True), (0, 400, 56, 64, 32, True)])
def test_dense_line(monkeypatch, problem, n, degree, graphs, B, dense):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the lines are shares of 152 SMs")
    import paper_2605_06921_gb300 as mq
    g = mi.erdos_renyi(n, degree / n, 1)
    G = mi.pack([g] * graphs) if graphs > 1 else g
    s = mq.Solver(mq.Graph(G), mq.params(problem=problem, batch=B, x_dtype=1))
    assert s.info()["dense"] == dense
