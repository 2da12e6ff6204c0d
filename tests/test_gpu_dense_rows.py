"""Which rows are summed apart from the tiles (long rows): the hubs of a graph, not the ordinary
rows of one whose agents all have many contacts, next to each other in one context; a graph's
forward then takes one launch a day, and both directions follow the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2207_09714_gb300 import capi, synth

from helpers import EXACT_MARGIN, check_adjoint, ensure_built, model, to_dev

pytestmark = pytest.mark.gpu

T, SEEDS = 40, 10


def graph(n, degree, hubs=0, seed=0):
    """Random pairs, `degree` a row on average; the first agents have 200, 300, ... contacts more."""
    rng = np.random.default_rng(seed)
    m = n * degree // 2
    u, v = [rng.integers(0, n, m)], [rng.integers(0, n, m)]
    for h in range(hubs):
        v.append(rng.choice(np.arange(hubs, n), 200 + 100 * h, replace=False))
        u.append(np.full(v[-1].size, h))
    u, v = np.concatenate(u), np.concatenate(v)
    return synth.csr_from_undirected(n, u, v, rng.uniform(0.5, 1.5, u.size), rng.integers(0, 9, n))


DENSE, HUBS = dict(n=2000, degree=110), dict(n=2500, degree=8, hubs=4, seed=1)


@pytest.mark.parametrize("policy", [capi.GABM_STORE_LAMBDA, capi.GABM_RECOMPUTE])
@pytest.mark.parametrize("specs,long_launches", [([DENSE], False), ([HUBS], True), ([DENSE, HUBS], True)],
                         ids=["dense", "hubs", "both"])
def test_hubs_are_long_rows_and_dense_rows_are_not(specs, long_launches, policy):
    ensure_built()
    pops = [graph(**s) for s in specs]
    I = len(pops)
    R, m = np.full((I, T), 2.6, np.float32), np.full((I, T), 0.02, np.float32)
    S = np.tile(synth.SUSCEPTIBILITY, (I, 1)).astype(np.float32)
    c = synth.infectiousness_table()
    for seed in range(32):   # a key without a near-tie: the trajectories must then be equal
        md_o = O.Model(4, 7, c, seed=seed)
        refs = [O.forward_hard(p, md_o, R[i], m[i], S[i], n_seed=SEEDS, inst=i) for i, p in enumerate(pops)]
        if min(r["margin"] for r in refs) > EXACT_MARGIN:
            break
    gD = np.stack([O.mse(r["D"], synth.target_curve(T, p.n, level=5e-5))[1] for r, p in zip(refs, pops)])
    ctx = capi.gabm_create(pops, model(c, seed=seed, policy=policy))
    dev = to_dev(R, m, S)
    before = capi.gabm_launch_count(ctx)
    capi.gabm_forward(ctx, T, *dev, [SEEDS] * I)
    launches = capi.gabm_launch_count(ctx) - before
    assert (launches >= 2 * T) == long_launches   # otherwise a launch a day and a dozen around them
    assert np.array_equal(capi.gabm_get_state(ctx)[0], np.concatenate([r["e_final"] for r in refs]))
    got = [x.cpu().numpy() for x in capi.gabm_backward(ctx, *to_dev(gD))]
    for i, p in enumerate(pops):
        want = O.backward_hard(p, md_o, R[i], m[i], S[i], refs[i]["e_final"], gD[i], inst=i)
        for k, v in zip(("dR", "dm", "dS"), got):
            check_adjoint(v[i], want[k], k)
