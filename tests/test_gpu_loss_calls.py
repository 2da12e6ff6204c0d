"""cumulative_mse is torch's own expression to its callers, whichever path it takes: what may be
done with the operands and the result of ((cumsum(D) - y) ** 2).mean() may be done with it."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def expression(D: torch.Tensor, y: torch.Tensor) -> torch.Tensor:
    return ((torch.cumsum(D, dim=-1) - y) ** 2).mean()


@pytest.fixture
def data():
    from helpers import ensure_built
    ensure_built()
    gen = torch.Generator(device="cuda").manual_seed(5)
    make = lambda: torch.rand((3, 70), generator=gen, dtype=torch.float64, device="cuda")
    return make(), torch.cumsum(make(), -1), make()


def loss_in_place(f, D, y, v):
    x = D.clone().requires_grad_()
    loss = f(x * 2.0, y)
    loss += 3.0
    loss *= 2.0
    return [loss.detach(), *torch.autograd.grad(loss, x)]


def operands_rewritten(f, D, y, v):
    x, y = D.clone().requires_grad_(), y.clone()
    d = x * 2.0
    loss = f(d, y)
    y.zero_()
    d.mul_(v)
    g, = torch.autograd.grad(loss, x, create_graph=True)
    h, = torch.autograd.grad((g * v).sum(), x)
    return [loss.detach(), g.detach(), h]


def target_made_in_inference_mode(f, D, y, v):
    with torch.inference_mode():
        y = y + 1.0
    x = D.clone().requires_grad_()
    loss = f(x, y)
    return [loss.detach(), *torch.autograd.grad(loss, x)]


def closed_over_by_a_transform(f, D, y, v):
    x = D.clone().requires_grad_()
    out = torch.func.vmap(lambda s: s * f(x, y))(v[:, 0])
    return [out.detach(), *torch.autograd.grad(out.sum(), x)]


def traced_symbolically(f, D, y, v):
    return [torch.fx.symbolic_trace(lambda d: f(d, y))(D)]


def traced_by_a_mode(f, D, y, v):
    from torch.fx.experimental.proxy_tensor import make_fx
    return [make_fx(lambda d: f(d, y))(D)(v)]


def scripted(f, D, y, v):
    return [torch.jit.script(f)(D, y)]


def batched_gradients(f, D, y, v):
    x = D.clone().requires_grad_()
    loss = f(x, y)
    return [torch.autograd.grad(loss, x, v[:, 0], is_grads_batched=True)[0]]


def without_a_graph(f, D, y, v):
    with torch.inference_mode():
        return [f(D, y).clone()]


USES = (loss_in_place, operands_rewritten, target_made_in_inference_mode, closed_over_by_a_transform,
        traced_symbolically, traced_by_a_mode, scripted, batched_gradients, without_a_graph)


@pytest.mark.parametrize("use", USES, ids=lambda u: u.__name__)
def test_used_as_the_torch_expression(use, data):
    from paper_2207_09714_gb300.calibrate import cumulative_mse
    got, want = use(cumulative_mse, *data), use(expression, *data)
    assert len(got) == len(want) > 0
    for a, b in zip(got, want):   # float64 sums of 210 terms: 1e-12 of the largest is far above rounding
        assert a.shape == b.shape and torch.all((a - b).abs() <= 1e-12 * b.abs().max())
