"""log_l1_loss under torch.jit.script, torch.jit.trace and torch.fx (CPU: the
tensor operations)."""
import pytest


@pytest.fixture(scope="module")
def A():
    import paper_2305_02678_gb300.autograd as A
    return A


def _inputs():
    import torch
    g = torch.Generator().manual_seed(0)
    return torch.randn((50, 3), generator=g), torch.rand((50, 3), generator=g)


@pytest.mark.filterwarnings("ignore::DeprecationWarning", "ignore::torch.jit.TracerWarning")
@pytest.mark.parametrize("how", ["script", "trace", "fx"])
def test_compiled_forms(A, how):
    import torch
    x, y = _inputs()
    f = {"script": lambda: torch.jit.script(A.log_l1_loss), "trace": lambda: torch.jit.trace(A.log_l1_loss, (x, y)),
         "fx": lambda: torch.fx.symbolic_trace(A.log_l1_loss)}[how]()
    a, b = x.clone().requires_grad_(), x.clone().requires_grad_()
    la, lb = f(a, y), A._log_l1_ops(b, y)
    la.backward()
    lb.backward()
    torch.testing.assert_close(la, lb)
    torch.testing.assert_close(a.grad, b.grad)
