"""Rows of more than 64 entries are summed apart from the SELL slices (a block each): graphs
whose rows sit at the edges of that rule -- 63 to 65 entries, one round of a block (512), a
remainder after it -- against the oracle, symmetric (in- and out-rows alike) and directed."""
import numpy as np
import pytest

import oracle as O
from paper_2207_09714_gb300 import capi, synth

from helpers import check_adjoint, ensure_built, model, to_dev

pytestmark = pytest.mark.gpu

T = 24
HUBS = (63, 64, 65, 128, 129, 511, 512, 513, 1500)


def hub_graph(directed, seed=0, n=2500):
    """Agent h of the first len(HUBS) is joined to HUBS[h] others; the rest meet at random."""
    rng = np.random.default_rng(seed)
    dst, src = [], []
    for h, k in enumerate(HUBS):
        others = rng.choice(np.arange(len(HUBS), n), size=k, replace=False)
        dst.append(np.full(k, h)); src.append(others)
    m = 3 * n
    dst.append(rng.integers(len(HUBS), n, m)); src.append(rng.integers(len(HUBS), n, m))
    dst, src = np.concatenate(dst), np.concatenate(src)
    age = rng.integers(0, 9, n)
    if not directed:
        return synth.csr_from_undirected(n, dst, src, rng.uniform(0.5, 1.5, dst.size), age)
    key = np.unique(dst * n + src)
    rowptr = np.zeros(n + 1, np.uint64)
    rowptr[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    return synth.Population(n=n, rowptr=rowptr, col=(key % n).astype(np.uint32), age=age.astype(np.uint8),
                            w=rng.uniform(0.5, 1.5, key.size).astype(np.float32))


@pytest.mark.parametrize("policy", [capi.GABM_STORE_LAMBDA, capi.GABM_RECOMPUTE])
@pytest.mark.parametrize("directed", [False, True])
def test_long_rows_follow_the_oracle(directed, policy):
    ensure_built()
    pop = hub_graph(directed)
    R = np.full((1, T), 2.6, np.float32)
    m = np.full((1, T), 0.02, np.float32)
    S = synth.SUSCEPTIBILITY[None, :].astype(np.float32)
    c = synth.infectiousness_table()
    y = synth.target_curve(T, pop.n, level=5e-5)[None, :]
    for seed in range(32):   # a key without a near-tie: the trajectories must then be equal
        md_o = O.Model(4, 7, c, seed=seed)
        ref = O.forward_hard(pop, md_o, R[0], m[0], S[0], n_seed=10)
        if ref["margin"] > 1e-6:
            break
    _, gD = O.mse(ref["D"], y[0])
    want = O.backward_hard(pop, md_o, R[0], m[0], S[0], ref["e_final"], gD)
    ctx = capi.gabm_create([pop], model(c, seed=seed, policy=policy))
    dev = to_dev(R, m, S)
    capi.gabm_forward(ctx, T, *dev, [10])
    assert np.array_equal(capi.gabm_get_state(ctx)[0], ref["e_final"])
    t = 12
    start = np.where((ref["e_final"] < t), ref["e_final"], capi.GABM_NEVER)
    day = O.day_hard(pop, md_o, t, float(R[0, t]), S[0], start)
    sus = start == capi.GABM_NEVER
    lam = float(R[0, t]) * S[0][pop.age].astype(np.float64) * day["Lam"]
    got = capi.gabm_get_lambda(ctx, t)[0].astype(np.float64)
    assert np.all(np.abs(got[sus] - lam[sus]) <= 1e-5 * np.abs(lam[sus]))
    dR, dm, dS, dc = capi.gabm_backward_table(ctx, to_dev(gD[None, :])[0])
    for k, v in (("dR", dR), ("dm", dm), ("dS", dS), ("dc", dc)):
        if k in want:
            check_adjoint(v.cpu().numpy()[0], want[k], k)
