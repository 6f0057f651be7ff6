"""f_B's backward under saved-tensor hooks that give the saved tensors back in
another layout, at another address or from host memory: the same gradient."""
import pytest

import mqo_inputs as mi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def offset(t):
    """the same values one element behind a 16-byte boundary"""
    base = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    base[1:] = t.reshape(-1)
    return base[1:].view(t.shape)


HOOKS = {
    "transposed": (lambda t: t.t().contiguous(), lambda t: t.t()),
    "offset": (lambda t: t, offset),
    "host": (lambda t: t.cpu(), lambda t: t.cuda()),
}


@pytest.mark.parametrize("hooks", list(HOOKS))
@pytest.mark.parametrize("B", [1, 4, 64])
def test_gradient_under_saved_tensor_hooks(hooks, B):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_2605_06921_gb300 as mq
    G = mi.chung_lu(3001, 2.5, 8.0, 3)
    g = mq.Graph(G)
    x = torch.rand((G.n, B), device="cuda", generator=torch.Generator("cuda").manual_seed(B)) * 2 - 1
    x.requires_grad_(True)
    gout = torch.linspace(0.5, 1.5, B, dtype=torch.float64, device="cuda")
    mq.FbObjective.apply(x, g, 0.001).backward(gout)
    want, x.grad = x.grad, None
    with torch.autograd.graph.saved_tensors_hooks(*HOOKS[hooks]):
        out = mq.FbObjective.apply(x, g, 0.001)
    out.backward(gout)
    assert torch.equal(x.grad, want)
