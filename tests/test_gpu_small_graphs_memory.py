"""Device memory of a context of many small graphs, per day of its horizon: beside the hazards, the
per-tile sums and some words an instance, what the sums of a day are reduced through grows with
the tiles, not with the graphs."""
import numpy as np
import pytest

import oracle as O
from paper_2207_09714_gb300 import capi, synth

from helpers import EXACT_MARGIN, check_adjoint, ensure_built, model, to_dev

pytestmark = pytest.mark.gpu


def held(pops, T):
    I = len(pops)
    ctx = capi.gabm_create(pops, model(seed=2))
    R, m = np.full((I, T), 2.5, np.float32), np.full((I, T), 0.02, np.float32)
    capi.gabm_forward(ctx, T, *to_dev(R, m, np.tile(synth.SUSCEPTIBILITY, (I, 1)).astype(np.float32)), [2] * I)
    got = capi.gabm_mem_stats(ctx)[0]
    capi.gabm_destroy(ctx)
    return got


@pytest.mark.parametrize("n", [30, 90])
def test_a_day_of_many_small_graphs(n):
    ensure_built()
    pops = [synth.population_small(n=n, seed=1)] * 600
    per_day = (held(pops, 512) - held(pops, 64)) / (512 - 64) / len(pops)
    tiles = -(-n // 32)
    # a tile: lambda, nine sums (FP64), the bitmap; an instance: D, gD, y, dR, dm, R, m, counts,
    # newRM twice, three scale words, Q -- and one more Q to reduce through
    assert per_day <= tiles * (128 + 72 + 4) + (5 * 8 + 2 * 4 + 6 * 4 + 3 * 4 + 72) + 72 + 2


@pytest.mark.parametrize("sizes", [(20,), (33, 20, 400), (3000, 20, 20)])
def test_gradients_of_small_graphs(sizes):
    """Few tiles a graph on average, so one share each, or two, or more."""
    ensure_built()
    T, seeds = 30, 5
    pops = [synth.population_small(n=n, seed=i) for i, n in enumerate(sizes)]
    I = len(pops)
    R, m = np.full((I, T), 2.8, np.float32), np.full((I, T), 0.05, np.float32)
    S = np.tile(synth.SUSCEPTIBILITY, (I, 1)).astype(np.float32)
    c = synth.infectiousness_table()
    for seed in range(40):   # a key without a near-tie: the trajectories must then be equal
        md = O.Model(4, 7, c, seed=seed)
        refs = [O.forward_hard(p, md, R[i], m[i], S[i], n_seed=seeds, inst=i) for i, p in enumerate(pops)]
        if min(r["margin"] for r in refs) > EXACT_MARGIN:
            break
    gD = np.stack([O.mse(r["D"], synth.target_curve(T, p.n, level=5e-5))[1] for r, p in zip(refs, pops)])
    ctx = capi.gabm_create(pops, model(c, seed=seed))
    capi.gabm_forward(ctx, T, *to_dev(R, m, S), [seeds] * I)
    got = [x.cpu().numpy() for x in capi.gabm_backward(ctx, *to_dev(gD))]
    for i, p in enumerate(pops):
        want = O.backward_hard(p, md, R[i], m[i], S[i], refs[i]["e_final"], gD[i], inst=i)
        for k, v in zip(("dR", "dm", "dS"), got):
            check_adjoint(v[i], want[k], k)
