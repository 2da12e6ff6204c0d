"""A graph whose long rows are of one direction only launches nothing for the other, and counts
nothing: directed weights, recomputed hazards, a few agents that many others hear of."""
import numpy as np
import pytest

from paper_2207_09714_gb300 import capi, synth

from helpers import ensure_built, model, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hubs_hear", [False, True], ids=["out-hubs", "in-hubs"])
def test_launches_of_a_reverse_day(hubs_hear):
    ensure_built()
    n, T = 2000, 40
    rng = np.random.default_rng(3)
    hub, other = np.repeat(np.arange(4), 300), np.concatenate([rng.choice(np.arange(4, n), 300, replace=False) for _ in range(4)])
    dst, src = rng.integers(4, n, 6 * n), rng.integers(4, n, 6 * n)
    key = np.unique(np.concatenate([dst, hub if hubs_hear else other]) * n + np.concatenate([src, other if hubs_hear else hub]))
    rowptr = np.zeros(n + 1, np.uint64)
    rowptr[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    pop = synth.Population(n=n, rowptr=rowptr, col=(key % n).astype(np.uint32), age=rng.integers(0, 9, n).astype(np.uint8),
                           w=rng.uniform(0.5, 1.5, key.size).astype(np.float32))
    ctx = capi.gabm_create([pop], model(seed=1, policy=capi.GABM_RECOMPUTE))
    R, m = np.full((1, T), 2.5, np.float32), np.full((1, T), 0.02, np.float32)
    capi.gabm_forward(ctx, T, *to_dev(R, m, synth.SUSCEPTIBILITY[None, :].astype(np.float32)), [20])
    before = capi.gabm_launch_count(ctx)
    capi.gabm_backward(ctx, *to_dev(np.ones((1, T))))
    # a day: the hazards, the sweep, and one launch of the long rows; less than a dozen around them
    assert capi.gabm_launch_count(ctx) - before < 3 * T + 12
