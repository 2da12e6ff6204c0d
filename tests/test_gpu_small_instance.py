"""Graphs of up to sixteen 32-row tiles per SM run the day kernels' small instances: a graph
of exactly that many tiles and one of a tile more (the larger instances, its last tile of one
row), in both directions, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_2207_09714_gb300 import capi, synth

from helpers import check_adjoint, ensure_built, model, to_dev

pytestmark = pytest.mark.gpu

T = 26


@pytest.mark.parametrize("extra", [0, 1])
def test_each_side_of_the_small_instances_line(extra):
    ensure_built()
    import torch
    n = 16 * 32 * torch.cuda.get_device_properties(0).multi_processor_count + extra
    rng = np.random.default_rng(extra)
    pop = synth.csr_from_undirected(n, rng.integers(0, n, 4 * n), rng.integers(0, n, 4 * n),
                                    rng.uniform(0.5, 1.5, 4 * n), rng.integers(0, 9, n))
    R = np.full((1, T), 2.6, np.float32)
    m = np.full((1, T), 0.02, np.float32)
    S = synth.SUSCEPTIBILITY[None, :].astype(np.float32)
    c = synth.infectiousness_table()
    for seed in range(32):   # a key without a near-tie: the trajectories must then be equal
        md_o = O.Model(4, 7, c, seed=seed)
        ref = O.forward_hard(pop, md_o, R[0], m[0], S[0], n_seed=60)
        if ref["margin"] > 1e-6:
            break
    _, gD = O.mse(ref["D"], synth.target_curve(T, n, level=5e-5))
    want = O.backward_hard(pop, md_o, R[0], m[0], S[0], ref["e_final"], gD)
    ctx = capi.gabm_create([pop], model(c, seed=seed))
    capi.gabm_forward(ctx, T, *to_dev(R, m, S), [60])
    assert np.array_equal(capi.gabm_get_state(ctx)[0], ref["e_final"])
    for k, v in zip(("dR", "dm", "dS"), capi.gabm_backward(ctx, to_dev(gD[None, :])[0])):
        check_adjoint(v.cpu().numpy()[0], want[k], k)
