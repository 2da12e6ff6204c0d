"""The autotuner called after a forward alone, before any loss gradient is known, times reverse
sweeps that have work to do: their days take about as long as a real backward's."""
import numpy as np
import pytest

from paper_2207_09714_gb300 import capi, synth

from helpers import ensure_built, model, to_dev

pytestmark = pytest.mark.gpu


def test_backward_schedules_are_timed_on_days_with_an_adjoint():
    ensure_built()
    B, T, n = 2, 60, 120_000   # two sets: one backward schedule, the one the backward below has too
    rng = np.random.default_rng(1)
    pop = synth.csr_from_undirected(n, rng.integers(0, n, 10 * n), rng.integers(0, n, 10 * n),
                                    rng.uniform(0.5, 1.5, 10 * n), rng.integers(0, 9, n))
    R, m = np.full((B, T), 2.5, np.float32), np.full((B, T), 0.02, np.float32)
    dev = to_dev(R, m, np.tile(synth.SUSCEPTIBILITY, (B, 1)).astype(np.float32))
    ctx = capi.gabm_create([pop], model(seed=2), sets_per_graph=B)
    capi.gabm_forward(ctx, T, *dev, [50] * B)

    def reverse_day(run):
        run()
        capi.gabm_set_profiling(ctx, True)
        run()
        ms, launches = capi.gabm_get_profile(ctx, 1)
        capi.gabm_set_profiling(ctx, False)
        return ms / launches

    tuned = reverse_day(lambda: capi.gabm_autotune(ctx, 3))
    (gD,) = to_dev(np.ones((B, T)))
    real = reverse_day(lambda: [capi.gabm_backward(ctx, gD) for _ in range(3)])
    assert tuned > 0.7 * real, (tuned, real)   # without an adjoint: a third or less
