"""The recomputing reverse sweep takes r and the hazard in one pass over a row's entries: its
gradients are bitwise those of the stored hazards, for rows of 1 to 30 entries (each side of a
batch of pairs), days with and without an adjoint, and the table's adjoint beside it."""
import numpy as np
import pytest

from paper_2207_09714_gb300 import capi, synth

from helpers import ensure_built, model, to_dev

pytestmark = pytest.mark.gpu

T = 32


def graph(n=6000):
    """Agent i draws 1 + i mod 15 partners nearby: rows of 1 to about 30 entries."""
    rng = np.random.default_rng(4)
    u = np.repeat(np.arange(n), 1 + np.arange(n) % 15)
    v = (u + rng.integers(1, 200, u.size)) % n
    return synth.csr_from_undirected(n, u, v, rng.uniform(0.5, 1.5, u.size), rng.integers(0, 9, n))


@pytest.mark.parametrize("last_loss_day", [T - 1, 20, 12])
@pytest.mark.parametrize("table", [False, True])
def test_recomputed_sweep_is_bitwise_the_stored_one(table, last_loss_day):
    ensure_built()
    pop = graph()
    R, m = np.full((1, T), 2.8, np.float32), np.full((1, T), 0.02, np.float32)
    dev = to_dev(R, m, synth.SUSCEPTIBILITY[None, :].astype(np.float32))
    gD = np.where(np.arange(T) <= last_loss_day, np.linspace(-1.0, 1.5, T), 0.0)[None, :]
    got = []
    for policy in (capi.GABM_STORE_LAMBDA, capi.GABM_RECOMPUTE):
        ctx = capi.gabm_create([pop], model(seed=8, policy=policy))
        capi.gabm_forward(ctx, T, *dev, [25])
        out = (capi.gabm_backward_table if table else capi.gabm_backward)(ctx, *to_dev(gD))
        got.append([x.cpu().numpy() for x in out])
    assert np.abs(got[0][0]).max() > 0
    for a, b in zip(*got):
        assert np.array_equal(a, b)
