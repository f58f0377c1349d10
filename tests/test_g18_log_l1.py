"""The one-pass log-L1 loss against the same loss in tensor operations:
value, derivative and second derivative, and the inputs that must keep going
through the tensor operations."""
import pytest

pytestmark = pytest.mark.gpu


def _inputs(n, seed=0):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn((n, 3), generator=g, device="cuda") * 2
    y = torch.rand((n, 3), generator=g, device="cuda") * 4
    x[0] = 0.0
    if n > 2:
        x[1], y[1] = y[1], y[1].clone()  # equal: sign(0)
        x[2, 0] = -0.0
    return x, y


@pytest.mark.parametrize("n", [1, 85, 86, 341, 342, 50000, 400001])
def test_value_and_gradient(n):
    import torch
    from paper_2305_02678_gb300 import autograd as A
    x, y = _inputs(n)
    a, b = x.clone().requires_grad_(), x.clone().requires_grad_()
    assert A._one_pass(a, y)
    l1, l2 = A.log_l1_loss(a, y), A._log_l1_ops(b.double(), y.double())
    assert l1.shape == () and l1.dtype == torch.float32
    # each value's error is a few roundings of its terms, which are positive
    assert abs(l1.item() - l2.item()) <= 1e-6 * l2.item()
    (3.0 * l1).backward()
    A._log_l1_ops(b, y).mul(3.0).backward()
    # three roundings on either side
    torch.testing.assert_close(a.grad, b.grad, rtol=4e-7, atol=0.0)
    assert A.log_l1_loss(a, y).item() == l1.item()  # a fixed order of summation
    with torch.no_grad():
        assert A.log_l1_loss(x, y).item() == l1.item()


def test_non_finite_values():
    import torch
    from paper_2305_02678_gb300 import autograd as A
    inf, nan = float("inf"), float("nan")
    x = torch.tensor([inf, -inf, nan, 1.0, 1.0, -1.0, 0.0, inf, -3.0, 2.0], device="cuda")
    y = torch.tensor([1.0, 1.0, 1.0, nan, inf, nan, nan, inf, -2.0, -1.0], device="cuda")
    a, b = x.clone().requires_grad_(), x.clone().requires_grad_()
    la, lb = A.log_l1_loss(a, y), A._log_l1_ops(b, y)
    la.backward()
    lb.backward()
    torch.testing.assert_close(la, lb, equal_nan=True, rtol=0, atol=0)
    torch.testing.assert_close(a.grad, b.grad, equal_nan=True, rtol=4e-7, atol=0)


def test_second_derivative_hooks_and_in_place_changes():
    import torch
    from paper_2305_02678_gb300 import autograd as A
    x, y = _inputs(100, 1)
    out = []
    for f in (A.log_l1_loss, A._log_l1_ops):
        a = x.clone().requires_grad_()
        h = a * 1.5
        g, = torch.autograd.grad(f(h, y) * 2.0, a, create_graph=True)
        g2, = torch.autograd.grad((g ** 2).sum(), a)
        out.append((g.detach(), g2))
    torch.testing.assert_close(out[0], out[1], rtol=1e-6, atol=0.0)
    a = x.clone().requires_grad_()
    seen = []
    with torch.autograd.graph.saved_tensors_hooks(lambda t: seen.append(t) or t.cpu(), lambda t: t.cuda()):
        l = A.log_l1_loss(a, y)
    assert seen
    with torch.no_grad():
        a.clamp_(min=0)  # the first derivative needs none of the inputs
    l.backward()
    b = x.clone().requires_grad_()
    A._log_l1_ops(b, y).backward()
    torch.testing.assert_close(a.grad, b.grad, rtol=4e-7, atol=0.0)


def test_other_inputs_keep_the_tensor_operations():
    import torch
    import torch.autograd.forward_ad as fwd_ad
    from paper_2305_02678_gb300 import autograd as A
    x, y = _inputs(64, 2)
    assert not A._one_pass(x.cpu(), y.cpu())
    assert not A._one_pass(x.double(), y.double())
    assert not A._one_pass(x.t(), y.t())
    assert not A._one_pass(x, y[:1])
    assert not A._one_pass(x, y.clone().requires_grad_())
    assert not A._one_pass(x[:0], y[:0])
    ref = A._log_l1_ops(x, y)
    per = torch.vmap(A.log_l1_loss)(x, y)
    torch.testing.assert_close(per.mean(), ref)
    g = torch.func.grad(A.log_l1_loss)(x, y)
    b = x.clone().requires_grad_()
    A._log_l1_ops(b, y).backward()
    torch.testing.assert_close(g, b.grad)
    with fwd_ad.dual_level():
        t = fwd_ad.unpack_dual(A.log_l1_loss(fwd_ad.make_dual(x, torch.ones_like(x)), y)).tangent
    torch.testing.assert_close(t, b.grad.sum())
    yt = y.clone().requires_grad_()
    A.log_l1_loss(x, yt).backward()
    assert yt.grad is not None


def test_under_graph_capture():
    import torch
    from paper_2305_02678_gb300 import autograd as A
    x, y = _inputs(5000, 3)
    out = torch.empty((), device="cuda")
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s), torch.no_grad():
        out.copy_(A.log_l1_loss(x, y))
    torch.cuda.current_stream().wait_stream(s)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph), torch.no_grad():
        out.copy_(A.log_l1_loss(x, y))
    x.mul_(0.5)
    graph.replay()
    assert out.item() == A.log_l1_loss(x, y).item()
