"""f_B under torch.compile: the graph breaks at the library's calls, the
objective and the gradient are those of the plain call."""
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("backend", ["eager", "aot_eager"])
@pytest.mark.parametrize("B", [4, 32])
def test_compiled_objective(backend, B):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2605_06921_gb300 as mq
    G = mi.chung_lu(2001, 2.5, 8.0, 3)
    g = mq.Graph(G)
    x = torch.rand((G.n, B), device="cuda", generator=torch.Generator("cuda").manual_seed(B)) * 2 - 1

    def loss(x):
        return (mq.FbObjective.apply(x * 0.5, g, 0.001) * 2.0).sum()

    torch._dynamo.reset()
    out = []
    for fn in (loss, torch.compile(loss, backend=backend)):
        y = x.clone().requires_grad_(True)
        v = fn(y)
        v.backward()
        with torch.no_grad():
            w = fn(y)
        assert not w.requires_grad
        out.append((v.detach(), w, y.grad))
    torch._dynamo.reset()
    (v0, w0, g0), (v1, w1, g1) = out
    # double sums of the same float32 terms in another order
    for a in (w0, v1, w1):
        assert torch.allclose(a, v0, rtol=1e-12, atol=1e-9)
    assert torch.equal(g0, g1)
