"""The reverse sweep keeps more of each row in flight (six pairs of entries a lane) where a
graph's rows, size and locality allow it: graphs on each side of that rule -- near and far
neighbours, short and long rows, rows around the twelve entries of one batch -- with stored
and recomputed hazards, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2207_09714_gb300 import capi, synth

from helpers import check_adjoint, ensure_built, model, to_dev

pytestmark = pytest.mark.gpu

T, N = 24, 150_000   # 150k agents: as many waves of tiles with either instance


def graph(near, degree):
    rng = np.random.default_rng(degree)
    m = N * degree // 2
    u = rng.integers(0, N, m)
    v = np.minimum(u + rng.integers(1, 40, m), N - 1) if near else rng.integers(0, N, m)
    return synth.csr_from_undirected(N, u, v, rng.uniform(0.5, 1.5, m), rng.integers(0, 9, N))


@pytest.mark.parametrize("policy", [capi.GABM_STORE_LAMBDA, capi.GABM_RECOMPUTE])
@pytest.mark.parametrize("near,degree", [(True, 6), (True, 12), (False, 12), (False, 25)])
def test_reverse_sweep_follows_the_oracle(near, degree, policy):
    ensure_built()
    pop = graph(near, degree)
    R = np.full((1, T), 2.6, np.float32)
    m = np.full((1, T), 0.02, np.float32)
    S = synth.SUSCEPTIBILITY[None, :].astype(np.float32)
    c = synth.infectiousness_table()
    for seed in range(64):   # a key without a near-tie: the trajectories must then be equal
        md_o = O.Model(4, 7, c, seed=seed)
        ref = O.forward_hard(pop, md_o, R[0], m[0], S[0], n_seed=60)
        if ref["margin"] > 1e-6:
            break
    _, gD = O.mse(ref["D"], synth.target_curve(T, N, level=5e-5))
    want = O.backward_hard(pop, md_o, R[0], m[0], S[0], ref["e_final"], gD)
    ctx = capi.gabm_create([pop], model(c, seed=seed, policy=policy))
    capi.gabm_forward(ctx, T, *to_dev(R, m, S), [60])
    assert np.array_equal(capi.gabm_get_state(ctx)[0], ref["e_final"])
    for k, v in zip(("dR", "dm", "dS"), capi.gabm_backward(ctx, to_dev(gD[None, :])[0])):
        check_adjoint(v.cpu().numpy()[0], want[k], k)
