"""Which step kernel member graphs that fit in shared memory take.  MaxCut: the
row groups while there are few items or short rows, the shared-memory kernel
beyond the measured line, whatever the storage type.  Few items: the staged
kernel, unless an item has little to gather or float32 rows are long."""
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("xd,vd", [(1, 1), (1, 0), (2, 2)])
@pytest.mark.parametrize("graphs,B,degree,kernel", [
    (64, 32, 6, "rows"), (64, 32, 32, "smem_wide"), (64, 64, 10, "rows"), (64, 64, 32, "smem_wide"),
    (64, 128, 20, "rows"), (64, 128, 60, "smem_wide"),
    (50, 32, 24, "rows"), (50, 32, 48, "smem_wide"), (50, 64, 36, "rows"), (50, 64, 60, "smem_wide"),
    (50, 128, 60, "rows"), (36, 32, 60, "smem_wide"), (36, 64, 60, "rows"),
    # rows too few to cover the latency of the longest one: not the row groups
    (36, 32, 36, "smem_wide")])
def test_rows_or_shared_memory(monkeypatch, graphs, B, degree, kernel, xd, vd):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the lines are shares of 152 SMs")
    import paper_2605_06921_gb300 as mq
    monkeypatch.setenv("MQO_TICK_KERNEL", "ticks")
    g = mi.erdos_renyi(400, degree / 400, 1)
    s = mq.Solver(mq.Graph(mi.pack([g] * graphs)), mq.params(problem=1, batch=B, x_dtype=xd, v_dtype=vd))
    assert s.info()["step_kernel"] == kernel


@pytest.mark.parametrize("problem", [0, 1])
@pytest.mark.parametrize("n,graphs,degree,B,xd,staged", [  # staged: MIS, MaxCut
    (60, 33, 10, 32, 1, (False, False)), (60, 33, 10, 32, 0, (False, False)), (30, 48, 4, 128, 1, (False, False)),
    (30, 48, 4, 128, 0, (True, True)), (30, 16, 4, 128, 1, (True, True)), (100, 16, 4, 32, 2, (False, True)),
    (60, 16, 4, 64, 1, (False, True)), (250, 8, 10, 32, 1, (True, True)), (250, 8, 10, 64, 0, (True, True)),
    (250, 48, 30, 64, 0, (False, False)), (60, 48, 30, 128, 0, (False, False)), (250, 16, 30, 64, 0, (True, True))])
def test_few_items(monkeypatch, problem, n, graphs, degree, B, xd, staged):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the lines are shares of 152 SMs")
    import paper_2605_06921_gb300 as mq
    monkeypatch.setenv("MQO_TICK_KERNEL", "ticks")
    g = mi.erdos_renyi(n, degree / n, 1)
    s = mq.Solver(mq.Graph(mi.pack([g] * graphs)), mq.params(problem=problem, batch=B, x_dtype=xd))
    assert (not s.info()["step_kernel"].startswith("smem")) == staged[problem]
