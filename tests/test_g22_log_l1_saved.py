"""What the one-pass log-L1 loss keeps for its derivatives: copies of its own,
held by the graph as saved tensors and by nothing else."""
import pytest

pytestmark = pytest.mark.gpu


def _inputs(n=1000, seed=0):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((n, 3), generator=g, device="cuda") * 2, torch.rand((n, 3), generator=g, device="cuda") * 4


def test_targets_made_in_inference_mode():
    import torch
    from paper_2305_02678_gb300 import autograd as A
    x, y = _inputs()
    with torch.inference_mode():
        target = y * 1.0
    a, b = x.clone().requires_grad_(), x.clone().requires_grad_()
    assert A._one_pass(a, target)
    A.log_l1_loss(a, target).backward()
    A._log_l1_ops(b, target).backward()
    torch.testing.assert_close(a.grad, b.grad, rtol=4e-7, atol=0.0)
    with torch.inference_mode():
        assert A.log_l1_loss(x * 1.0, target).item() == A.log_l1_loss(x, y).item()


def test_second_and_third_derivative_after_the_inputs_changed():
    import torch
    from paper_2305_02678_gb300 import autograd as A
    x, y = _inputs(100)
    x[0], x[1, 0], x[1, 1] = 0.0, -1.0, 99.0
    out = []
    for f in (A.log_l1_loss, A._log_l1_ops):
        a, t = x.clone().requires_grad_(), y.clone()
        h = a * 1.5
        l = f(h, t)
        with torch.no_grad():
            h.zero_()
            t.fill_(7.0)
        w = torch.tensor(2.0, device="cuda", requires_grad=True)
        g, = torch.autograd.grad(l * w, a, create_graph=True)
        g2, gw = torch.autograd.grad((g ** 2).sum(), (a, w), create_graph=True)
        g3, = torch.autograd.grad((g2 * g2).sum(), a)
        out.append([v.detach() for v in (g, g2, gw, g3)])
    for p, q in zip(*out):
        # a handful of roundings each, and FP32 sums of 300 positive terms
        torch.testing.assert_close(p, q, rtol=5e-6, atol=0.0)


@pytest.mark.parametrize("second", [False, True])
def test_nothing_outlives_the_backward(second):
    import torch
    from paper_2305_02678_gb300 import autograd as A
    n = 200000
    leaf, y = _inputs(n)
    leaf.requires_grad_()
    A.log_l1_loss(leaf * 1.0, y).backward()
    leaf.grad = None
    torch.cuda.synchronize()
    base = torch.cuda.memory_allocated()
    losses = []
    for _ in range(3):
        losses.append(A.log_l1_loss(leaf * 1.0, y.clone()))
        if second:
            g, = torch.autograd.grad(losses[-1], leaf, create_graph=True)
            (g ** 2).sum().backward()
            del g
        else:
            losses[-1].backward()
        leaf.grad = None
    assert torch.cuda.memory_allocated() - base < n  # three scalars; a tensor is 12 n


def test_hooks_see_everything_saved():
    import torch
    from paper_2305_02678_gb300 import autograd as A
    x, y = _inputs()
    x.requires_grad_()
    torch.cuda.synchronize()
    with torch.autograd.graph.saved_tensors_hooks(lambda t: t.cpu(), lambda t: t.cuda()):
        before = torch.cuda.memory_allocated()
        h = x * 1.0
        one = torch.cuda.memory_allocated() - before
        l = A.log_l1_loss(h, y)
        del h
    assert torch.cuda.memory_allocated() - before <= one  # the scalar; all else is on the host
    g, = torch.autograd.grad(l, x, create_graph=True)
    assert g.requires_grad and torch.isfinite(g).all()


@pytest.mark.parametrize("n_work", [1, 7, 304, 1000])
def test_no_more_blocks_than_the_workspace_holds(n_work):
    import torch
    from paper_2305_02678_gb300 import autograd as A
    from paper_2305_02678_gb300 import binding as B
    x, y = _inputs(100000)
    loss = torch.zeros((), device="cuda")
    work = torch.full((n_work + 400,), -5.0, dtype=torch.float64, device="cuda")
    B._check(B.lib().nam_internal_log_l1(x.data_ptr(), y.data_ptr(), x.numel(), None, None, loss.data_ptr(),
                                         work.data_ptr(), n_work, B.current_stream(x.device)), "log_l1")
    assert (work[n_work:] == -5.0).all()
    # FP32 sums of up to 300,000 / 256 positive terms in a thread
    assert abs(loss.item() - A._log_l1_ops(x.double(), y.double()).item()) <= 1200 * 2.0 ** -24 * loss.item()
