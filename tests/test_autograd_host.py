"""The gradients of GabmFunction are tensors of their own: one may be written in place, or kept,
without the others (a stand-in for the library's calls; no GPU)."""
import pytest
import torch

from paper_2207_09714_gb300 import capi
from paper_2207_09714_gb300.autograd import GabmFunction

I, T, A = 2, 6, capi.GABM_NUM_AGES


@pytest.fixture
def gradients(monkeypatch):
    def backward(ctx, gD, *out):
        out = out or [torch.empty(s, dtype=torch.float64) for s in ((I, T), (I, T), (I, A))]
        for k, x in enumerate(out):
            x.copy_(gD.sum() * (k + 1.0) + torch.arange(x.numel(), dtype=torch.float64).reshape(x.shape))
        return tuple(out)

    monkeypatch.setattr(capi, "gabm_forward", lambda ctx, T, R, m, S, n_seed: (torch.ones(I, T, dtype=torch.float64), None))
    monkeypatch.setattr(capi, "gabm_backward", backward)
    leaves = [torch.rand(s, requires_grad=True) for s in ((I, T), (I, T), (I, A))]
    D = GabmFunction.apply(object(), *leaves, [3, 4])
    return torch.autograd.grad(D.sum(), leaves)


def test_writing_one_gradient_leaves_what_was_built_from_another(gradients):
    dR, dm, dS = gradients
    w = torch.full_like(dR, 2.0, requires_grad=True)
    q = (dR * w).sum()
    before = dR.clone()
    dm.zero_()
    dS.mul_(3.0)
    q.backward()
    assert torch.equal(w.grad, before)


def test_each_gradient_holds_its_own_memory(gradients):
    for g, shape in zip(gradients, ((I, T), (I, T), (I, A))):
        assert g.shape == shape and g.dtype == torch.float32 and g._base is None
        assert g.untyped_storage().nbytes() == g.numel() * g.element_size()
