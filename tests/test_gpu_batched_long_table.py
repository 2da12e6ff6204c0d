"""The table adjoint of many sets holds L x sets sums a warp in shared memory: tables on either
side of the 48 KB a block has without asking for more (64 sets: L = 14, 20), and the longest."""
import numpy as np
import pytest

import oracle as O
from paper_2207_09714_gb300 import capi, synth

from helpers import EXACT_MARGIN, check_adjoint, ensure_built, model, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau_IR", [9, 10, 16, 28])
def test_table_adjoint_of_64_sets(tau_IR):
    ensure_built()
    B, T, n_seed = 64, 40, 12
    pop = synth.population_small(n=1500, seed=7)
    c = synth.infectiousness_table(4, tau_IR)
    rng = np.random.default_rng(tau_IR)
    R = rng.uniform(2.0, 3.5, (B, 1)) * rng.uniform(0.9, 1.1, (B, T))
    R, m = R.astype(np.float32), np.full((B, T), 0.02, np.float32)
    S = np.tile(synth.SUSCEPTIBILITY, (B, 1)).astype(np.float32)
    ctx = capi.gabm_create([pop], model(c, 4, tau_IR, seed=9), sets_per_graph=B)
    dev = to_dev(R, m, S)
    capi.gabm_forward(ctx, T, *dev, [n_seed] * B)
    md_o = O.Model(4, tau_IR, c, seed=9)
    refs = [O.forward_hard(pop, md_o, R[i], m[i], S[i], n_seed=n_seed, inst=i) for i in range(B)]
    gD = np.stack([O.mse(r["D"], synth.target_curve(T, pop.n, level=5e-5))[1] for r in refs])
    got = [x.cpu().numpy() for x in capi.gabm_backward_table(ctx, *to_dev(gD))]
    exact = [i for i in range(B) if refs[i]["margin"] > EXACT_MARGIN]
    assert len(exact) >= 8
    for i in exact:
        want = O.backward_hard(pop, md_o, R[i], m[i], S[i], refs[i]["e_final"], gD[i], inst=i)
        for k, v in zip(("dR", "dm", "dS"), got):
            check_adjoint(v[i], want[k], k)
        check_adjoint(got[3][i][1:], want["dc"][1:], "dc")
