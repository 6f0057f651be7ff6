"""The shared-memory limit of a kernel is the same whatever the solver that
launches it: host threads with solvers of different sizes would otherwise
lower it between each other's setting and launch."""
import pytest

import cudart_shim

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CODE = """
import os
import mqo_inputs as mi
import paper_2605_06921_gb300 as mq
# step kernel, discrete kernel, ticks: one solver each of two sizes
for env, kw, sizes, p, want in [
        (dict(MQO_TICK_KERNEL="small"), dict(batch=4), (60, 200), 0.1, dict(small=True)),
        (dict(MQO_STEP_KERNEL="dense"), dict(batch=32, x_dtype=1), (300, 1000), 0.3, dict(dense=True)),
        (dict(MQO_STEP_KERNEL="staged"), dict(batch=32, x_dtype=1), (60, 300), 0.5, dict(step_kernel="staged")),
        (dict(MQO_STEP_KERNEL="smem"), dict(batch=32, x_dtype=1), (60, 300), 0.1, dict(step_kernel="smem", ell=False)),
        (dict(MQO_STEP_ELL="1"), dict(batch=32, x_dtype=1), [(60,) * 200, (300,) * 200], 0.1, dict(ell=True)),
        (dict(MQO_STEP_ELL="1", MQO_STEP_KERNEL="wide"), dict(batch=32), [(60,) * 200, (300,) * 200], 0.1,
         dict(ell=True, step_kernel="smem_wide")),
        (dict(MQO_DISC_KERNEL="graph"), dict(batch=32), (60, 300), 0.1, dict(discrete_kernel="graph")),
        (dict(MQO_DISC_KERNEL="bits"), dict(batch=32), (300, 600), 0.3, dict(discrete_kernel="graph"))]:
    os.environ.setdefault("MQO_TICK_KERNEL", "ticks")
    os.environ.update(env)
    for n in sizes:
        G = mi.pack([mi.erdos_renyi(m, p, m) for m in n]) if isinstance(n, tuple) else mi.erdos_renyi(n, p, n)
        s = mq.Solver(mq.Graph(G), mq.params(**kw))
        info = s.info()
        assert all(info[k] == v for k, v in want.items()), (env, info)
        s.run(17)
        s.step(1)
        s.best()
    for k in set(env) | {"MQO_TICK_KERNEL"}:
        os.environ.pop(k)
"""


def test_limit_of_a_kernel_does_not_depend_on_the_solver(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    log = tmp_path / "attributes"
    cudart_shim.run(tmp_path, CODE, SHIM_ATTR_LOG=str(log))
    limits = {}
    for line in log.read_text().splitlines():
        kernel, attribute, value = line.split()
        if attribute == "8":  # cudaFuncAttributeMaxDynamicSharedMemorySize
            limits.setdefault(kernel, set()).add(int(value))
    assert len(limits) >= 8
    assert all(len(v) == 1 for v in limits.values()), limits
