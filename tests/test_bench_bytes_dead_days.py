"""The bench's byte counts of the reverse days as the kernels run them: an exposure that can die
only after the horizon has no adjoint, nor has anything it would cause, so the coefficients
of those days are 0 (in the oracle's sweep as well); rows gather nothing from such a day and
its ring slot is neither written nor read.  Counted row by row here (no GPU)."""
import os
import sys

import numpy as np
import pytest

import oracle as O
from paper_2207_09714_gb300 import synth

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

NEVER, T, L = 32767, 26, 11


def trajectory(n=500, seed=1):
    pop = synth.population_small(n=n, seed=seed)
    R, m = np.full(T, 2.8, np.float32), np.full(T, 0.05, np.float32)
    S = synth.SUSCEPTIBILITY.astype(np.float32)
    md = O.Model(4, 7, synth.infectiousness_table(), seed=seed)
    ref = O.forward_hard(pop, md, R, m, S, n_seed=12)
    return pop, md, R, m, S, ref


@pytest.mark.parametrize("store", [True, False])
def test_reverse_days_as_a_per_row_count(store):
    pop, _, _, _, _, ref = trajectory()
    E, deg = ref["e_final"].astype(np.int64), np.diff(pop.rowptr.astype(np.int64))
    n_rows = (pop.n + 31) // 32 * 32
    last = bench.last_counting_day(T, L)
    got = bench.trajectory_bytes(E, deg.astype(np.float64), T, L, n_rows, store, last=last)[1]
    for t in range(T):
        want = 6.0 * n_rows + 36.0 * (n_rows // 32)
        slots = [t + k for k in range(2, L) if t + k <= last]
        for e, d in zip(E, deg):
            seed, never = e < 0, e == NEVER
            if t + 1 <= last and not seed and e >= t + 2 - L:
                want += 8.0 * d + 4.0
            if not seed and e >= t:
                want += 1.0 + 4.0 * len(slots) + 4.0 + (4.0 if store else 0.0) + (0.0 if never else 4.0)
        assert got[t] == want, t


def test_no_coefficient_after_the_last_counting_day():
    pop, md, R, m, S, ref = trajectory()
    _, gD = O.mse(ref["D"], synth.target_curve(T, pop.n, level=5e-5))
    last = bench.last_counting_day(T, L)
    g = O.backward_hard(pop, md, R, m, S, ref["e_final"], gD)
    assert np.all(g["dR"][last + 1:] == 0.0) and g["dR"][last] != 0.0
