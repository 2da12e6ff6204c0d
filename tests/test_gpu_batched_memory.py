"""Device memory of a context with several sets per graph, per day of its horizon: the stored
hazards (32 rows x sets floats a tile) and, for the gradients' partial sums, no more than a whole
tile's nine age bins in FP64 would take -- whatever part of a tile a warp works on."""
import numpy as np
import pytest

from paper_2207_09714_gb300 import capi, synth

from helpers import ensure_built, model, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [5, 16, 64])
def test_a_day_takes_no_more_than_whole_tiles_would(B):
    ensure_built()
    pop = synth.population_small(n=4000, seed=3)
    ntiles, Bp = -(-pop.n // 32), 1 << (B - 1).bit_length()
    held = []
    for T in (64, 512):
        ctx = capi.gabm_create([pop], model(seed=1), sets_per_graph=B)
        R, m = np.full((B, T), 2.5, np.float32), np.full((B, T), 0.01, np.float32)
        S = np.tile(synth.SUSCEPTIBILITY, (B, 1)).astype(np.float32)
        capi.gabm_forward(ctx, T, *to_dev(R, m, S), [10] * B)
        held.append(capi.gabm_mem_stats(ctx)[0])
        capi.gabm_destroy(ctx)
    per_day = (held[1] - held[0]) / (512 - 64)
    whole_tiles = ntiles * Bp * (32 * 4 + 9 * 8)
    assert per_day <= whole_tiles + 256 * B   # and some words a set: deaths, counts, parameters, gradients
