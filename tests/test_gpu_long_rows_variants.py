"""Long rows (more than 64 entries) of both directions -- agents with many in-contacts, other
agents with many out-contacts -- in every variant of the model, in contexts of several graphs
and in a forward resumed from a set state, against each variant's oracle."""
import numpy as np
import pytest

import oracle as O
from oracle import durations as DU
from oracle import fate as F
from oracle import sirs as SI
from paper_2207_09714_gb300 import capi, synth

from helpers import EXACT_MARGIN, check_adjoint, ensure_built, model, to_dev

pytestmark = pytest.mark.gpu

T, SEEDS = 30, 60
IN_HUBS, OUT_HUBS = (64, 65, 130, 600), (65, 66, 128, 513, 900)
PMF = np.array([0.1, 0.2, 0.3, 0.15, 0.1, 0.1, 0.05], np.float32)
S = synth.SUSCEPTIBILITY.astype(np.float32)


def hub_graph(seed=0, n=2400):
    """Directed: the first agents hear from 64 to 600 others, the next are heard by 65 to 900."""
    rng = np.random.default_rng(seed)
    a, b = len(IN_HUBS), len(IN_HUBS) + len(OUT_HUBS)
    dst, src = [rng.integers(b, n, 3 * n)], [rng.integers(b, n, 3 * n)]
    for h, k in enumerate(IN_HUBS):
        dst.append(np.full(k, h)); src.append(rng.choice(np.arange(b, n), k, replace=False))
    for h, k in enumerate(OUT_HUBS):
        src.append(np.full(k, a + h)); dst.append(rng.choice(np.arange(b, n), k, replace=False))
        dst.append(np.full(30, a + h)); src.append(rng.choice(np.arange(b, n), 30, replace=False))
    key = np.unique(np.concatenate(dst) * n + np.concatenate(src))
    rowptr = np.zeros(n + 1, np.uint64)
    rowptr[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    return synth.Population(n=n, rowptr=rowptr, col=(key % n).astype(np.uint32),
                            age=rng.integers(0, 9, n).astype(np.uint8),
                            w=rng.uniform(0.5, 1.5, key.size).astype(np.float32))


def params(instances, seed=0):
    rng = np.random.default_rng(seed)
    return (rng.uniform(3.0, 4.0, (instances, T)).astype(np.float32),
            rng.uniform(0.05, 0.2, (instances, T)).astype(np.float32), np.tile(S, (instances, 1)))


def variant(name, seed):
    """(model of the library, run of the oracle -> forward, adjoint of a gD)."""
    c = synth.infectiousness_table()
    if name == "sirs":
        mo = SI.SirsModel(4, 7, 6, c, seed=seed)
        return (capi.ModelDesc(4, 7, c, seed=seed, tau_RS=6), lambda *a, **k: SI.forward(a[0], mo, *a[1:], **k),
                lambda p, R, m, f, gD: SI.backward(p, mo, R, m, S, f["e_hist"], gD))
    if name == "fate":
        c = synth.infectiousness_table(4, 10)
        mo = F.FateModel(4, 7, 10, c, seed=seed)
        return (capi.ModelDesc(4, 7, c, seed=seed, tau_IM=10), lambda *a, **k: F.forward(a[0], mo, *a[1:], **k),
                lambda p, R, m, f, gD: F.backward(p, mo, R, m, S, f["e_final"], gD))
    if name == "durations":
        mo = DU.DurationModel(4, 7, PMF, c, seed=seed)
        return (capi.ModelDesc(4, 7, c, seed=seed, p_IR=PMF), lambda *a, **k: DU.forward(a[0], mo, *a[1:], **k),
                lambda p, R, m, f, gD: DU.backward(p, mo, R, m, S, f["e_final"], gD))
    mo = O.Model(4, 7, c, seed=seed)
    policy = capi.GABM_RECOMPUTE if name == "recompute" else capi.GABM_STORE_LAMBDA
    return (model(c, seed=seed, policy=policy), lambda *a, **k: O.forward_hard(a[0], mo, *a[1:], **k),
            lambda p, R, m, f, gD, inst=0: O.backward_hard(p, mo, R, m, S, f["e_final"], gD, inst=inst))


def exact_key(name, run):
    """A key without a near-tie draw: the trajectories must then be equal."""
    for seed in range(40):
        md, fwd, bwd = variant(name, seed)
        fs = run(fwd)
        if min(f["margin"] for f in fs) > EXACT_MARGIN:
            return md, bwd, fs
    raise AssertionError("no key without a near-tie")


def loss_gradient(f, p):
    return O.mse(f["D"], synth.target_curve(T, p.n, seed=2, level=5e-5))[1]


@pytest.mark.parametrize("name", ["store", "recompute", "sirs", "fate", "durations"])
def test_variant_follows_its_oracle(name):
    ensure_built()
    pop = hub_graph()
    R, m, Sd = params(1)
    md, bwd, (f,) = exact_key(name, lambda fwd: [fwd(pop, R[0], m[0], S, n_seed=SEEDS)])
    hubs = slice(len(IN_HUBS), len(IN_HUBS) + len(OUT_HUBS))
    assert (f["e_final"][hubs] < capi.GABM_NEVER).sum() >= 2   # hubs among the infectious
    gD = loss_gradient(f, pop)
    want = bwd(pop, R[0], m[0], f, gD)
    ctx = capi.gabm_create([pop], md)
    D, counts = capi.gabm_forward(ctx, T, *to_dev(R, m, Sd), [SEEDS], want_counts=True)
    assert np.array_equal(capi.gabm_get_state(ctx)[0].astype(np.int64), f["e_final"])
    assert np.array_equal(counts.cpu().numpy()[0], f["counts"])
    assert np.allclose(D.cpu().numpy()[0], f["D"], rtol=1e-15, atol=0)
    base = name in ("store", "recompute")
    got = (capi.gabm_backward_table if base else capi.gabm_backward)(ctx, *to_dev(gD[None, :]))
    for k, v in zip(("dR", "dm", "dS"), got):
        check_adjoint(v.cpu().numpy()[0], want[k], k)
    if base:
        check_adjoint(got[3].cpu().numpy()[0][1:], want["dc"][1:], "dc")


def test_soft_relaxation_follows_its_oracle():
    ensure_built()
    pop = hub_graph()
    R, m, Sd = params(1)
    c = synth.infectiousness_table()
    md = O.Model(4, 7, c, seed=3)
    f = O.forward_soft(pop, md, R[0], m[0], S, n_seed=SEEDS)
    gD = loss_gradient(f, pop)
    want = O.backward_soft(pop, md, R[0], m[0], S, gD, f["s_hist"], f["y_hist"], f["dydl_hist"], f["Lam_hist"], f["newRM"])
    ctx = capi.gabm_create([pop], capi.ModelDesc(4, 7, c, seed=3, relax_mode=capi.GABM_SOFT))
    D, _ = capi.gabm_forward(ctx, T, *to_dev(R, m, Sd), [SEEDS])
    assert np.allclose(D.cpu().numpy()[0], f["D"], rtol=1e-4, atol=1e-6 * np.abs(f["D"]).max())
    for k, v in zip(("dR", "dm", "dS"), capi.gabm_backward(ctx, *to_dev(gD[None, :]))):
        check_adjoint(v.cpu().numpy()[0], want[k], k)


@pytest.mark.parametrize("name", ["store", "recompute"])
def test_two_graphs_with_hubs_in_one_context(name):
    ensure_built()
    pops = [hub_graph(0), hub_graph(1, 1700)]
    R, m, Sd = params(2, 5)
    R[1, 12:] = 0.0   # the second graph's late days carry no adjoint, the first one's do
    md, bwd, fs = exact_key(name, lambda fwd: [fwd(p, R[i], m[i], S, n_seed=SEEDS, inst=i) for i, p in enumerate(pops)])
    gD = np.stack([loss_gradient(f, p) for f, p in zip(fs, pops)])
    ctx = capi.gabm_create(pops, md)
    capi.gabm_forward(ctx, T, *to_dev(R, m, Sd), [SEEDS] * 2)
    assert np.array_equal(capi.gabm_get_state(ctx)[0], np.concatenate([f["e_final"] for f in fs]))
    got = [x.cpu().numpy() for x in capi.gabm_backward(ctx, *to_dev(gD))]
    for i, p in enumerate(pops):
        want = bwd(p, R[i], m[i], fs[i], gD[i], inst=i)
        for k, v in zip(("dR", "dm", "dS"), got):
            check_adjoint(v[i], want[k], k)


@pytest.mark.parametrize("day", [1, 9, 20])
def test_forward_resumed_from_a_set_state(day):
    ensure_built()
    pop = hub_graph()
    R, m, Sd = params(1)
    md, bwd, (f,) = exact_key("recompute", lambda fwd: [fwd(pop, R[0], m[0], S, n_seed=SEEDS)])
    start = np.where(f["e_final"] < day, f["e_final"], capi.GABM_NEVER).astype(np.int16)
    ctx = capi.gabm_create([pop], md)
    capi.gabm_set_state(ctx, day, start[None, :])
    capi.gabm_forward(ctx, T, *to_dev(R, m, Sd))
    assert np.array_equal(capi.gabm_get_state(ctx)[0], f["e_final"])
    gD = loss_gradient(f, pop)
    want = bwd(pop, R[0], m[0], f, gD)
    for k, v in zip(("dR", "dm", "dS"), capi.gabm_backward(ctx, *to_dev(gD[None, :]))):
        check_adjoint(v.cpu().numpy()[0], want[k], k)
