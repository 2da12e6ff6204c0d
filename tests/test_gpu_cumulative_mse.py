"""The fused cumulative-death loss against the torch expression it stands for, at the edges of a
block's piece of days (256), with its gradient's gradient."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1), (1, 255), (3, 256), (64, 257), (2, 700)])
def test_cumulative_mse_matches_torch(shape):
    import torch
    from helpers import ensure_built
    from paper_2207_09714_gb300.calibrate import cumulative_mse
    ensure_built()
    gen = torch.Generator(device="cuda").manual_seed(shape[1])
    D, y, v = (torch.rand(shape, generator=gen, dtype=torch.float64, device="cuda") for _ in range(3))
    y = torch.cumsum(y, -1)
    plain = lambda x: ((torch.cumsum(x, -1) - y) ** 2).mean()
    got, want = [], []
    for f, out in ((lambda x: cumulative_mse(x, y), got), (plain, want)):
        x = D.clone().requires_grad_()
        loss = f(x)
        g, = torch.autograd.grad(loss, x, create_graph=True)
        h, = torch.autograd.grad((g * v).sum(), x)
        x2 = D.clone().requires_grad_()
        f(x2).mul(3.0).backward()
        out += [loss.detach(), g.detach(), h, x2.grad]
    # sums of up to 64 x 700 positive or mixed float64 terms: 1e-12 of the largest is far above rounding
    for a, b in zip(got, want):
        assert torch.all((a - b).abs() <= 1e-12 * b.abs().max())
