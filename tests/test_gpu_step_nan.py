"""Steps of MIS from an x with values that are no numbers, or out of the box:
every step kernel gives the global-memory kernel's iterate, rounding and exact
counts (a NaN is not in the set, and hides no neighbour that is)."""
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

DT = {0: torch.float32, 1: torch.bfloat16, 2: torch.float16}
PLANS = {
    "staged": (dict(MQO_STEP_KERNEL="staged"), lambda i: i["step_kernel"] == "staged"),
    "smem": (dict(MQO_STEP_KERNEL="smem"), lambda i: i["step_kernel"] == "smem" and not i["ell"]),
    "wide": (dict(MQO_STEP_KERNEL="wide"), lambda i: i["step_kernel"] == "smem_wide" and not i["ell"]),
    "ell": (dict(MQO_STEP_KERNEL="smem", MQO_STEP_ELL="1"), lambda i: i["step_kernel"] == "smem" and i["ell"]),
    "wide_ell": (dict(MQO_STEP_KERNEL="wide", MQO_STEP_ELL="1"), lambda i: i["step_kernel"] == "smem_wide" and i["ell"]),
    "rows": (dict(MQO_STEP_KERNEL="rows"), lambda i: i["step_kernel"] == "rows"),
    "dense": (dict(MQO_STEP_KERNEL="dense"), lambda i: i["dense"]),
    "small": (dict(MQO_TICK_KERNEL="small"), lambda i: i["small"]),
}


def step(mq, monkeypatch, env, ok, G, x0, **kw):
    with monkeypatch.context() as m:
        for k, v in dict(dict(MQO_TICK_KERNEL="ticks"), **env).items():
            m.setenv(k, v)
        s = mq.Solver(mq.Graph(G), mq.params(**kw))
    if not ok(s.info()):
        return None
    s.set_x(x0)
    s.step(1)
    return [s.get_x(), s.get_v(), s.round(), *s.step_stats()]


@pytest.mark.parametrize("B,xd", [(16, 1), (16, 2), (32, 0), (32, 1), (32, 2), (64, 1), (128, 2)])
@pytest.mark.parametrize("share", [0.01, 0.3])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -0.5, 3.0])
def test_irregular_x(monkeypatch, B, xd, share, value):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2605_06921_gb300 as mq
    G = mi.pack([mi.erdos_renyi(n, 0.2, n) for n in (90, 33, 150)])
    gen = torch.Generator(device="cuda").manual_seed(B + xd)
    x0 = (torch.rand((G.n, B), device="cuda", generator=gen) < 0.1).float()
    x0[torch.rand(x0.shape, device="cuda", generator=gen) < share] = value
    x0 = x0.to(DT[xd])
    kw = dict(batch=B, x_dtype=xd, alpha=0.5, momentum=0.4)
    want = step(mq, monkeypatch, dict(MQO_STEP_KERNEL="generic"), lambda i: i["step_kernel"] == "global", G, x0, **kw)
    ran = 0
    for name, (env, ok) in PLANS.items():
        got = step(mq, monkeypatch, env, ok, G, x0, **kw)
        if got is None:
            continue
        ran += 1
        for a, b in zip(got, want):
            same = (a == b) | (torch.isnan(a) & torch.isnan(b)) if a.is_floating_point() else a == b
            assert bool(same.all()), name
    assert ran >= 2
