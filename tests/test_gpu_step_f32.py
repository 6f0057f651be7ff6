"""The shared-memory step kernel with the sliced-ELL stream for float32 x, and
for every type below 32 trajectories, against the plain global-memory kernel:
the same steps, statistics and bits, for rows of 0, 1 and many entries, items
of 1 to 256 rows, and x out of the box or not a number."""
import numpy as np
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


def packed():
    star = mi.from_edges(151, np.zeros(150, int), np.arange(1, 151))
    parts = [mi.erdos_renyi(1, 0.5, 0), mi.erdos_renyi(256, 0.3, 1), mi.erdos_renyi(257, 0.01, 2), star,
             mi.erdos_renyi(390, 0.15, 3)]
    return mi.pack(parts * 12)  # items enough for the shared-memory kernel


@pytest.mark.parametrize("problem,objective", [(0, 0), (1, 0), (1, 2)])
@pytest.mark.parametrize("B,xd,vd", [(b, 0, 0) for b in (4, 8, 16, 32, 64)]
                         + [(4, 1, 1), (8, 2, 2), (16, 1, 0), (16, 2, 0), (16, 1, 1), (4, 2, 0)])
@pytest.mark.parametrize("special", [None, float("nan"), float("inf"), -0.0, 1e-30])
def test_f32_step_equals_generic(mq, monkeypatch, problem, objective, B, xd, vd, special):
    monkeypatch.setenv("MQO_TICK_KERNEL", "ticks")
    G = packed()
    gen = torch.Generator(device="cuda").manual_seed(B)
    x0 = ((torch.rand((G.n, B), device="cuda", generator=gen) - 0.45) * 2.4).clamp(-problem, 1)
    if special is not None:
        x0[torch.rand(x0.shape, device="cuda", generator=gen) < 0.01] = special
    out = []
    for force in (None, "generic"):
        if force:
            monkeypatch.setenv("MQO_STEP_KERNEL", force)
        else:
            monkeypatch.delenv("MQO_STEP_KERNEL", raising=False)
        s = mq.Solver(mq.Graph(G), mq.params(problem=problem, objective=objective, batch=B, x_dtype=xd, v_dtype=vd,
                                             gamma=1.7, lambda_=0.3, alpha=0.8 if problem == 0 else 0.02, momentum=0.4))
        info = s.info()
        assert (info["step_kernel"], info["ell"]) == (("global", False) if force else ("smem_wide", True))
        s.set_x(x0.to([torch.float32, torch.bfloat16, torch.float16][xd]))
        s.step(1 if special is not None else 5)
        out.append([s.get_x(), s.get_v(), *s.step_stats(), s.round()])
    for p, q in zip(*out):
        if p.is_floating_point():
            assert bool(((p == q) | (torch.isnan(p) & torch.isnan(q))).all())
        else:
            assert torch.equal(p, q)


def test_f32_step_default_outside_shared_memory(mq, monkeypatch):
    """long steps of wide float32 rows read them from L2, short ones and narrow rows are staged; the same steps"""
    for name in ("MQO_STEP_KERNEL", "MQO_STEP_ELL", "MQO_COL16"):
        monkeypatch.delenv(name, raising=False)
    G = mq.Graph(mi.erdos_renyi(10000, 0.002, 1))
    out = []
    for B, force, kern in ((128, None, "global"), (128, "staged", "staged"), (64, None, "staged")):
        if force:
            monkeypatch.setenv("MQO_STEP_KERNEL", force)
        else:
            monkeypatch.delenv("MQO_STEP_KERNEL", raising=False)
        s = mq.Solver(G, mq.params(batch=B, seed=3))
        assert s.info()["step_kernel"] == kern
        s.init()
        s.step(3)
        out.append(s.get_x())
    assert torch.equal(out[0], out[1])
