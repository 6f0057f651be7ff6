"""The training step that gathers once (the forward keeps A X) against the two
separate passes, and the four-at-a-time optimiser kernels against the scalar
ones (taken off the 16-byte boundary) and the written formulas."""
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


def hub_graph(n, hub, seed):
    rng = np.random.default_rng(seed)
    u = np.concatenate([rng.integers(0, n, 4 * n), np.zeros(hub, dtype=np.int64)])
    v = np.concatenate([rng.integers(0, n, 4 * n), rng.permutation(n)[:hub]])
    return mi.from_edges(n, u, v)


@pytest.mark.parametrize("B", [1, 4, 16, 32, 64, 256])
@pytest.mark.parametrize("n,hub", [(5, 0), (700, 513), (4000, 3000)])
def test_gradient_from_kept_product(mq, B, n, hub):
    g = mq.Graph(hub_graph(n, hub, B))
    X = (torch.rand((n, B), device="cuda") * 2 - 1).requires_grad_(True)
    gout = torch.linspace(-1.0, 2.0, B, device="cuda", dtype=torch.float64)
    obj = mq.FbObjective.apply(X, g, 0.01)
    (obj * gout).sum().backward()
    assert torch.equal(X.grad, mq.spmm_grad(g, X.detach(), 0.01, gout))
    ref = mq.fb_forward(g, X.detach(), 0.01)
    # double sums of the same float32 terms in another order
    assert torch.allclose(obj.detach(), ref, rtol=1e-12, atol=1e-9)
    with torch.no_grad():
        assert not mq.FbObjective.apply(X, g, 0.01).requires_grad
    assert torch.allclose(mq.FbObjective.apply(X.detach(), g, 0.01), ref, rtol=1e-12, atol=1e-9)


def test_change_in_place_is_still_an_error(mq):
    g = mq.Graph(hub_graph(100, 0, 1))
    X = torch.zeros((100, 8), device="cuda", requires_grad=True)
    obj = mq.FbObjective.apply(X, g, 0.01).sum()
    with torch.no_grad():
        X.add_(1.0)
    with pytest.raises(RuntimeError, match="modified by an inplace operation"):
        obj.backward()


@pytest.mark.parametrize("n", [1, 3, 4, 1023, 1024, 4099])
@pytest.mark.parametrize("kind", ["momentum", "adam"])
def test_optimiser_four_at_a_time(mq, kind, n):
    gen = torch.Generator(device="cuda").manual_seed(n)
    out = []
    base = [torch.randn(n, device="cuda", generator=gen) for _ in range(4)]
    base[2] = base[2].abs()
    for off in (0, 1):  # off = 1: one float past a 16-byte boundary
        t = []
        for b in base:
            buf = torch.zeros(n + off, device="cuda")
            buf[off:] = b
            t.append(buf[off:])
        if kind == "momentum":
            mq.pga_momentum_step(t[0], t[1], t[3], 0.1, 0.9, -1.0, 1.0)
        else:
            mq.pga_adam_step(t[0], t[1], t[2], t[3], 0.1, 0.9, 0.999, 1e-8, 3, -1.0, 1.0)
        out.append([b.clone() for b in t])
    for a, b in zip(*out):
        assert torch.equal(a, b)
