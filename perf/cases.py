"""The calls a user of this framework waits for, as measurable cases.

A case is one forward run or one training step (forward, loss on the cumulative deaths,
straight-through adjoint) of the epidemic model on a synthetic contact graph, through the
package's public entry points.  Graphs, parameters and Philox keys come from the seed
alone and are made on the GPU; ``exact`` restates the model and its adjoint in 64-bit
torch.  The families:

* forecast   ``gabm_forward`` with stage counts, then ``gabm_get_state``: a what-if run;
* step       ``GabmFunction`` forward and backward: the step a calibration repeats;
* table      ``TableFunction``: the step that also learns the infectiousness table, which
             moves from one step to the next;
* locations  the step on an agent-location graph.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2207_09714_gb300 import autograd, calibrate, capi, synth

TAU_EI, TAU_IR = 4, 7          # the stage times of the repository's workloads
NEVER = 32767
HOUSEHOLD_P = 0.4              # geometric household sizes up to 6


def listed():
    return [
        # the repository's 10k-agent workload: one county town, a forward run of a month;
        # the smallest call, where launches and latency count
        case("forecast_10k", "forecast", 10_000, 30, contacts="small"),
        # the same town calibrated: the smallest training step
        case("step_10k", "step", 10_000, 30, contacts="small"),
        # a four-month forecast of a mid-sized county (an odd agent count), most of it infected by the end
        case("forecast_250k", "forecast", 250_007, 120),
        # the headline workload of the benchmark: 1M agents, 60 days, 20 seeds
        case("step_1m", "step", 1_000_000, 60),
        # hubs of a power-law contact graph under the recompute policy (no lambda store), 90 days
        case("step_powerlaw_300k", "step", 300_000, 90, contacts="powerlaw", recompute=True, seeds=60),
        # a joint calibration's simulator: twelve uneven counties in one context, own parameters each
        case("counties_12", "step", 35_000, 60, counties=12),
        # an ensemble of 64 parameter sets on one graph, 45 days (the benchmark's batched workload, smaller)
        case("sets_64", "step", 200_000, 45, sets=64),
        # a small ensemble with an odd set count (padded inside) on an odd-sized town
        case("sets_12", "step", 50_021, 60, sets=12),
        # two consecutive calibration steps that learn the infectiousness table
        case("table_100k", "table", 100_000, 60),
        # agents meeting at households, schools, workplaces and venues, two hops a day
        case("locations_300k", "locations", 300_000, 60),
        # reinfection ten days after recovery
        case("sirs_200k", "step", 200_000, 60, tau_RS=10),
        # a mortality stage of its own (deaths sampled)
        case("split_200k", "step", 200_000, 60, tau_IM=10),
    ]


def case(name, kind, n, days, sets=1, counties=1, contacts="typed", recompute=False, tau_IM=0, tau_RS=0, seeds=20):
    c = dict(kind=kind, n=n, days=days, sets=sets, counties=counties, contacts=contacts, recompute=recompute,
             tau_IM=tau_IM, tau_RS=tau_RS, seeds=seeds)
    return dict(c, name=name) if name else c


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    family = rng.choice(["small", "forecast", "step", "powerlaw", "counties", "sets", "table", "locations", "sirs", "split"])
    seeds = rng.randint(10, 60)
    if family == "small":
        return case(None, rng.choice(["forecast", "step"]), size(5_000, 25_000), rng.randint(20, 45), contacts="small", seeds=seeds)
    if family == "forecast":
        return case(None, "forecast", size(25_000, 400_000), rng.randint(30, 120), seeds=seeds)
    if family == "step":
        return case(None, "step", size(25_000, 800_000), rng.randint(30, 60), seeds=seeds)
    if family == "powerlaw":
        return case(None, "step", size(50_000, 300_000), rng.randint(45, 90), contacts="powerlaw", recompute=True, seeds=seeds)
    if family == "counties":
        g = rng.randint(3, 32)
        return case(None, "step", size(4_000, 400_000 // g), rng.randint(30, 60), counties=g, seeds=seeds)
    if family == "sets":
        b = rng.randint(3, 64)
        return case(None, "step", size(10_000, min(200_000, 8_000_000 // b)), rng.randint(25, 45), sets=b, seeds=seeds)
    if family == "table":
        return case(None, "table", size(20_000, 200_000), rng.randint(30, 60), seeds=seeds)
    if family == "locations":
        return case(None, "locations", size(30_000, 400_000), rng.randint(30, 60), seeds=seeds)
    if family == "sirs":
        return case(None, "step", size(30_000, 300_000), rng.randint(30, 60), tau_RS=rng.randint(6, 14), seeds=seeds)
    return case(None, "step", size(30_000, 300_000), rng.randint(30, 60), tau_IM=rng.choice([4, 7, 10]), seeds=seeds)


# --------------------------------------------------------------------------- graphs, made on the GPU
def _runs(sizes, total):
    """Group of each of `total` consecutive members, and each group's end, for random sizes cut to fit."""
    ends = torch.cumsum(sizes, 0)
    gid = torch.searchsorted(ends, torch.arange(total, device=sizes.device), right=True)
    return gid, torch.clamp(ends, max=total)


def _household_sizes(n, gen):
    p = torch.tensor([HOUSEHOLD_P * (1 - HOUSEHOLD_P) ** k for k in range(6)], device="cuda")
    return torch.multinomial(p, n, replacement=True, generator=gen) + 1


def _uniform_sizes(n, lo, hi, gen):
    return torch.randint(lo, hi + 1, (max(n // lo, 1) + 1,), generator=gen, device="cuda")


def _clique_pairs(members, sizes):
    """Every pair within consecutive groups of `members`."""
    n = members.numel()
    gid, ends = _runs(sizes, n)
    pos = torch.arange(n, device="cuda")
    later = ends[gid] - pos - 1                       # members of the group after this one
    u = torch.repeat_interleave(pos, later)
    first = torch.cumsum(later, 0) - later
    v = u + 1 + torch.arange(u.numel(), device="cuda") - first[u]
    return members[u], members[v]


def _contact_graph(n, contacts, gen):
    """Households and random contacts ("small"), or households, schools, workplaces and random
    contacts with typed weights ("typed"; "powerlaw": the random contacts have hubs)."""
    age = torch.randint(0, 9, (n,), generator=gen, device="cuda")
    typed = contacts != "small"
    hh = _household_sizes(n, gen) if typed else torch.randint(1, 7, (n,), generator=gen, device="cuda")
    parts = [_clique_pairs(torch.arange(n, device="cuda"), hh) + (synth.TYPE_WEIGHT["household"],)]
    if typed:
        for place, lo, hi in (("school", 0, 1), ("workplace", 2, 6)):
            who = torch.nonzero((age >= lo) & (age <= hi)).flatten()
            who = who[torch.randperm(who.numel(), generator=gen, device="cuda")]
            parts.append(_clique_pairs(who, _uniform_sizes(who.numel(), 5, 30, gen)) + (synth.TYPE_WEIGHT[place],))
    if contacts == "powerlaw":
        kk = torch.arange(1, 2001, dtype=torch.float64, device="cuda")
        want = kk[torch.multinomial(kk ** -2.5, n, replacement=True, generator=gen)]
        cdf = torch.cumsum(want, 0)
        ends = torch.rand((2, int(want.sum()) // 2), generator=gen, dtype=torch.float64, device="cuda") * cdf[-1]
        u, v = torch.clamp(torch.searchsorted(cdf, ends, right=True), max=n - 1)
    else:
        u, v = torch.randint(0, n, (2, n * (5 if typed else 10) // 2), generator=gen, device="cuda")
    parts.append((u, v, synth.TYPE_WEIGHT["random"]))
    u, v = (torch.cat([p[k] for p in parts]) for k in (0, 1))
    scale = torch.cat([torch.full(p[0].shape, p[2] if typed else 1.0, device="cuda") for p in parts])
    w = scale * (0.5 + torch.rand(u.numel(), generator=gen, device="cuda"))
    u, v = torch.minimum(u, v), torch.maximum(u, v)
    key = torch.cat([u * n + v, v * n + u])           # both directions; a pair met twice keeps its first weight
    key, order = torch.sort(key, stable=True)
    keep = torch.ones_like(key, dtype=torch.bool)
    keep[1:] = key[1:] != key[:-1]
    keep &= (key // n) != (key % n)
    key, w = key[keep], torch.cat([w, w])[order][keep]
    return SimpleNamespace(n=n, rowptr=_rowptr(key // n, n), col=key % n, w=w, age=age)


def _location_graph(n, gen):
    """One household per agent, a school or workplace by age, and about 1.5 of n/40 venues."""
    age = torch.randint(0, 9, (n,), generator=gen, device="cuda")
    agents, locs, scale, base = [], [], [], 0

    def attend(who, sizes, weight):
        nonlocal base
        gid, _ = _runs(sizes, who.numel())
        agents.append(who)
        locs.append(base + gid)
        scale.append(torch.full(who.shape, weight, device="cuda"))
        base += int(gid[-1]) + 1 if gid.numel() else 0

    attend(torch.arange(n, device="cuda"), _household_sizes(n, gen), synth.TYPE_WEIGHT["household"])
    for place, lo, hi, smin, smax in (("school", 0, 1, 100, 400), ("workplace", 2, 6, 5, 60)):
        who = torch.nonzero((age >= lo) & (age <= hi)).flatten()
        who = who[torch.randperm(who.numel(), generator=gen, device="cuda")]
        attend(who, _uniform_sizes(who.numel(), smin, smax, gen), synth.TYPE_WEIGHT[place])
    venues = max(1, n // 40)
    who = torch.randint(0, n, (n * 3 // 2,), generator=gen, device="cuda")
    agents.append(who)
    locs.append(base + torch.randint(0, venues, who.shape, generator=gen, device="cuda"))
    scale.append(torch.full(who.shape, synth.TYPE_WEIGHT["random"], device="cuda"))
    base += venues
    key, order = torch.sort(torch.cat(agents) * base + torch.cat(locs), stable=True)
    w = torch.cat(scale)[order] * (0.5 + torch.rand(key.numel(), generator=gen, device="cuda"))
    keep = torch.ones_like(key, dtype=torch.bool)
    keep[1:] = key[1:] != key[:-1]
    key, w = key[keep], w[keep]
    return SimpleNamespace(n=n, n_loc=base, rowptr=_rowptr(key // base, n), loc=key % base, w=w, age=age)


def _rowptr(rows, n):
    out = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    out[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return out


def _inputs(case, seed):
    """Graphs, parameters and targets of a case, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    rng = np.random.default_rng(int(seed))
    n, T, B, G = case["n"], case["days"], case["sets"], case["counties"]
    sizes = [n] if G == 1 else [max(64, int(n * f)) for f in np.exp(rng.uniform(np.log(0.25), np.log(2.0), G))]
    make = _location_graph if case["kind"] == "locations" else lambda k, g: _contact_graph(k, case["contacts"], g)
    graphs = [make(k, gen) for k in sizes]
    inst = G * B
    lo, hi = (1.8, 3.2) if inst > 1 else (2.4, 2.6)
    daily = rng.uniform(0.95, 1.05, (inst, T))         # R and m vary by instance and day
    R = rng.uniform(lo, hi, (inst, 1)) * daily
    m = rng.uniform(0.005, 0.02, (inst, 1)) * rng.uniform(0.9, 1.1, (inst, T))
    S = synth.SUSCEPTIBILITY[None, :] * rng.uniform(0.9, 1.1, (inst, 1))
    y = np.cumsum(2e-6 * np.repeat(sizes, B)[:, None] * np.exp(0.08 * np.arange(T))[None, :], axis=1)
    tau_IM = case["tau_IM"]
    c = synth.infectiousness_table(TAU_EI, max(TAU_IR, tau_IM))
    tables = [c]
    if case["kind"] == "table":                        # the table before and after an optimiser's step
        moved = c * rng.uniform(0.95, 1.05, c.size)
        tables.append((moved / moved.sum()).astype(np.float32))

    def put(a, dt=torch.float32):
        return torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()

    return SimpleNamespace(graphs=graphs, R=put(R), m=put(m), S=put(S), y=put(y, torch.float64), tables=tables,
                           key=int(rng.integers(1 << 40)), n_seed=[case["seeds"]] * inst)


# --------------------------------------------------------------------------- the measured calls
def prepare(case, seed):
    s = _inputs(case, seed)
    model = capi.ModelDesc(TAU_EI, TAU_IR, s.tables[0], seed=s.key, tau_IM=case["tau_IM"], tau_RS=case["tau_RS"],
                           lambda_policy=capi.GABM_RECOMPUTE if case["recompute"] else capi.GABM_STORE_LAMBDA)
    if case["kind"] == "locations":
        hosted = [SimpleNamespace(n=g.n, n_loc=g.n_loc, rowptr=g.rowptr.cpu().numpy(), loc=g.loc.cpu().numpy(),
                                  w=g.w.cpu().numpy(), age=g.age.cpu().numpy()) for g in s.graphs]
        ctx = capi.gabm_create_bipartite(hosted, model)
    else:
        held = [SimpleNamespace(n=g.n, rowptr=g.rowptr.view(torch.uint64), col=g.col.to(torch.int32).view(torch.uint32),
                                w=g.w, age=g.age.to(torch.uint8)) for g in s.graphs]
        ctx = capi.gabm_create(held, model, sets_per_graph=case["sets"])
    grad = case["kind"] != "forecast"
    leaves = [x.requires_grad_(grad) for x in (s.R, s.m, s.S)]
    tables = [torch.from_numpy(c).cuda().requires_grad_() for c in s.tables]
    return SimpleNamespace(kind=case["kind"], ctx=ctx, leaves=leaves, tables=tables, y=s.y, n_seed=s.n_seed)


def run(state):
    R, m, S = state.leaves
    if state.kind == "forecast":
        D, counts = capi.gabm_forward(state.ctx, R.shape[1], R, m, S, state.n_seed, want_counts=True)
        return {"D": D, "counts": counts, "state": capi.gabm_get_state(state.ctx, device=True)}
    if state.kind == "table":
        out = []
        for c in state.tables:
            D = calibrate.TableFunction.apply(state.ctx, R, m, S, c, state.n_seed)
            loss = calibrate.cumulative_mse(D, state.y)
            dR, dm, dS, dc = torch.autograd.grad(loss, (R, m, S, c))
            out.append({"D": D.detach(), "loss": loss.detach(), "dR": dR, "dm": dm, "dS": dS, "dc": dc})
        return out
    D = autograd.GabmFunction.apply(state.ctx, R, m, S, state.n_seed)
    loss = calibrate.cumulative_mse(D, state.y)
    dR, dm, dS = torch.autograd.grad(loss, (R, m, S))
    return {"D": D.detach(), "loss": loss.detach(), "dR": dR, "dm": dm, "dS": dS}


def work(case):
    """What a pass cannot do without.  Forward: the graph once and every agent's exposure day (2
    bytes) each day.  Backward: the graph once for each day with a later day's adjoint to carry
    back, and per agent and day the state, the force of infection and the coefficients it leaves."""
    agents = case["n"] if case["counties"] == 1 else case["n"] * case["counties"] * 0.84
    per = {"small": 13.3, "typed": 22.4, "powerlaw": 20.0}[case["contacts"]]
    if case["kind"] == "locations":
        per = 2 * 3.3                                  # two hops over the attendances
    edges, slots, T, L = agents * per, agents * case["sets"], case["days"], TAU_EI + max(TAU_IR, case["tau_IM"])
    steps = 2 if case["kind"] == "table" else 1
    nbytes, flops = 8 * edges + 2.0 * T * slots, 2.0 * edges * case["sets"]
    if case["kind"] != "forecast":
        days = max(1, T - L)
        nbytes += days * (8 * edges + 12.0 * slots)
        flops += days * 2.0 * edges * case["sets"]
    return {"bytes": steps * nbytes, "flops": steps * flops}


# --------------------------------------------------------------------------- 64-bit restatement
_LOW = 0xFFFFFFFF


def _word(key, ids, day, inst, stream):
    """First word of Philox4x32-10 at counter (id, day, instance, stream), in int64 arithmetic."""
    ids, inst = torch.broadcast_tensors(ids, inst)
    x = [ids, torch.full_like(ids, day), inst, torch.full_like(ids, stream)]
    k0, k1 = key & _LOW, key >> 32

    def mul(c, v):
        low, high = c * (v & 0xFFFF), c * (v >> 16)
        return (high + (low >> 16)) >> 16, (low + ((high & 0xFFFF) << 16)) & _LOW

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, x[0])
        h1, l1 = mul(0xCD9E8D57, x[2])
        x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & _LOW, (k1 + 0xBB67AE85) & _LOW
    return x[0]


def _uniform(key, ids, day, inst, stream):
    return ((_word(key, ids, day, inst, stream) >> 9).double() + 0.5) * 2.0 ** -23


def _csr(rowptr, col, w, shape):
    return torch.sparse_csr_tensor(rowptr, col, w.double(), size=shape)


def _pair_sums(g):
    """x -> sum_j W_ij x_j on the graph's pairs (all graphs here are symmetric), and the mean degree."""
    w = g.w.double()
    if not hasattr(g, "loc"):
        A = _csr(g.rowptr, g.col, w, (g.n, g.n))
        return (lambda x: A @ x), float(w.sum()) / g.n
    rows = torch.repeat_interleave(torch.arange(g.n, device="cuda"), g.rowptr.diff())
    order = torch.argsort(g.loc, stable=True)
    A = _csr(g.rowptr, g.loc, w, (g.n, g.n_loc))
    At = _csr(_rowptr(g.loc, g.n_loc), rows[order], w[order], (g.n_loc, g.n))
    own = torch.zeros(g.n, dtype=torch.float64, device="cuda").index_add_(0, rows, w * w)
    s1 = torch.zeros(g.n_loc, dtype=torch.float64, device="cuda").index_add_(0, g.loc, w)
    return (lambda x: A @ (At @ x) - own[:, None] * x), float((s1 * s1).sum() - own.sum()) / g.n


def _simulate(case, s, g, inst0, c):
    """Forward of one graph's sets: a dict of the trajectory, and what the adjoint reads of it."""
    T, B, cols = case["days"], case["sets"], slice(inst0, inst0 + case["sets"])
    L_R, L_M = TAU_EI + TAU_IR, TAU_EI + case["tau_IM"]
    fate, cycle = case["tau_IM"] > 0, (L_R + case["tau_RS"]) if case["tau_RS"] else 1 << 20
    c = torch.from_numpy(c).cuda().double()
    L = c.numel()
    pull, dbar = _pair_sums(g)
    R, m, S = (x[cols].double() for x in (s.R, s.m, s.S))
    ids = torch.arange(g.n, device="cuda")[:, None]
    inst = torch.arange(inst0, inst0 + B, device="cuda")[None, :]
    Sa = S.T[g.age]                                    # [n, B]
    e = torch.full((g.n, B), NEVER, device="cuda")
    order = torch.argsort(_word(s.key, ids, 0, inst, 1) * g.n + ids, dim=0)
    for b in range(B):
        e[order[: s.n_seed[inst0 + b], b], b] = -TAU_EI
    leave = torch.full_like(e, L_R)                    # days from exposure to leaving I
    mortal = torch.zeros_like(e, dtype=torch.bool)     # those who leave I into M
    if fate:
        mortal = (e != NEVER) & (_uniform(s.key, ids, 0, inst, 1) < m[:, 0])
        leave = torch.where(mortal, L_M, leave)
    days, D, counts, exits = [], [], [], []
    for t in range(T):
        k = t - e
        seen = e != NEVER
        sus = ~seen | (k >= cycle)
        x = torch.where(seen & (k >= 1) & (k < leave), c[k.clamp(0, L - 1)], 0.0)
        Lam = pull(x) / dbar
        u = _uniform(s.key, ids, t, inst, 0)
        lam = R[:, t] * Sa * Lam
        new = sus & (u < -torch.expm1(-lam))
        out = seen & ~sus & (k == leave)
        exits.append(out.sum(0))
        D.append((out & mortal).sum(0).double() if fate else m[:, t] * out.sum(0))
        inside = seen & ~sus
        counts.append(torch.stack([sus.sum(0), (inside & (k < TAU_EI)).sum(0), (inside & (k >= TAU_EI) & (k < leave)).sum(0),
                                   (inside & (k >= leave)).sum(0)], -1))
        days.append((e.to(torch.int16), sus if cycle < 1 << 20 else None, Lam, new))
        e = torch.where(new, t, e)
        if fate:
            dies = (_uniform(s.key, ids, t + TAU_EI, inst, 1) < m[:, t + TAU_EI]) if t + TAU_EI < T else torch.zeros_like(new)
            leave = torch.where(new, torch.where(dies, L_M, L_R), leave)
            mortal = torch.where(new, dies, mortal)
    return SimpleNamespace(days=days, e=e, D=torch.stack(D, 1), counts=torch.stack(counts, 1), exits=torch.stack(exits, 1),
                           pull=pull, dbar=dbar, Sa=Sa, R=R, m=m, S=S, c=c, ids=ids, inst=inst, L_R=L_R, L_M=L_M, fate=fate,
                           cycle=cycle, age=g.age)


def _adjoint(case, s, f, gD):
    """Straight-through adjoint of a simulated graph, given dL/dD [B, T]."""
    T, L, B = case["days"], f.c.numel(), gD.shape[0]
    shape = f.e.shape
    zero = torch.zeros(shape, dtype=torch.float64, device="cuda")
    gx, later = {}, {T: zero}                          # gx of day t + k; dL/ds(t) of days still needed
    r = zero
    dR, dm, dc = torch.zeros_like(f.R), torch.zeros_like(f.R), torch.zeros(B, L, dtype=torch.float64, device="cuda")
    dS = torch.zeros_like(f.S)
    L_min, sign = min(f.L_R, f.L_M), (1.0 if f.L_M > f.L_R else -1.0)
    for t in range(T - 1, -2, -1):
        gx[t + 1] = f.pull(r) if t + 1 < T else zero
        gx.pop(t + 1 + L, None)
        if case["kind"] == "table":                    # every exposure k days before t + 1
            for k in range(1, L):
                dc[:, k] += torch.where(f.e == t + 1 - k, gx[t + 1], 0.0).sum(0)
        if t < 0:
            break
        e, sus, Lam, new = f.days[t]
        if sus is None:
            sus = e == NEVER
        G = torch.zeros(shape, dtype=torch.float64, device="cuda")
        if f.fate:
            H = torch.zeros(shape, dtype=torch.float64, device="cuda")
            v = _uniform(s.key, f.ids, t + TAU_EI, f.inst, 1) if t + TAU_EI < T else zero
            dies = (v < f.m[:, t + TAU_EI]) if t + TAU_EI < T else torch.zeros_like(new)
            if t + f.L_M < T:
                G += torch.where(dies, gD[:, t + f.L_M], 0.0)
                H += gD[:, t + f.L_M]
            for k in range(1, min(L, T - t)):
                G += torch.where(k < torch.where(dies, f.L_M, f.L_R), f.c[k] * gx[t + k], 0.0)
                if k >= L_min:
                    H += sign * f.c[k] * gx[t + k]
            if t + TAU_EI < T:
                mi = f.m[:, t + TAU_EI]
                dm[:, t + TAU_EI] += torch.where(new, H * v * (1 - v) / (mi * (1 - v) + (1 - mi) * v) ** 2, 0.0).sum(0)
        else:
            if t + f.L_R < T:
                G += f.m[:, t + f.L_R] * gD[:, t + f.L_R]
            for k in range(1, min(L, T - t)):
                G += f.c[k] * gx[t + k]
            dm[:, t] = gD[:, t] * f.exits[:, t]
            if t + f.cycle <= T:
                G += later[t + f.cycle]
        dy = torch.where(sus, G - later[t + 1], 0.0)
        later[t] = torch.where(new, G, later[t + 1])
        if f.cycle >= 1 << 20:
            later.pop(t + 1)
        u = _uniform(s.key, f.ids, t, f.inst, 0)
        lam = f.R[:, t] * f.Sa * Lam
        q, p = torch.exp(-lam), -torch.expm1(-lam)
        gl = dy * u * (1 - u) * q / (p * (1 - u) + q * u) ** 2
        dR[:, t] = (f.Sa * gl * Lam).sum(0)
        dS += torch.zeros_like(f.S.T).index_add_(0, f.age, f.R[:, t] * gl * Lam).T
        r = f.R[:, t] * f.Sa * gl / f.dbar
    if f.fate:                                         # the seeds drew their fate on day 0
        v, mi = _uniform(s.key, f.ids, 0, f.inst, 1), f.m[:, 0]
        H = zero + (gD[:, f.L_M - TAU_EI] if f.L_M - TAU_EI < T else 0.0)
        for k in range(max(L_min, TAU_EI), min(L, T + TAU_EI)):
            H = H + sign * f.c[k] * gx[k - TAU_EI]
        seed = f.days[0][0] != NEVER
        dm[:, 0] += torch.where(seed, H * v * (1 - v) / (mi * (1 - v) + (1 - mi) * v) ** 2, 0.0).sum(0)
    return dR, dm, dS, dc


def exact(case, seed):
    if case["n"] * case["sets"] * case["counties"] * case["days"] > 1_200_000_000:
        return None                                    # would take longer than it is worth
    s = _inputs(case, seed)
    results = []
    for c in s.tables:
        sims = [_simulate(case, s, g, i * case["sets"], c) for i, g in enumerate(s.graphs)]
        D = torch.cat([f.D for f in sims])
        if case["kind"] == "forecast":
            return {"D": D, "counts": None, "state": None}
        Dg = D.clone().requires_grad_()
        loss = ((torch.cumsum(Dg, -1) - s.y) ** 2).mean()
        gD, = torch.autograd.grad(loss, Dg)
        B = case["sets"]
        grads = [_adjoint(case, s, f, gD[i * B:(i + 1) * B]) for i, f in enumerate(sims)]
        dR, dm, dS, dc = (torch.cat(x) for x in zip(*grads))
        out = {"D": D, "loss": loss.detach(), "dR": dR, "dm": dm, "dS": dS}
        if case["kind"] == "table":
            out["dc"] = dc.sum(0)
        results.append(out)
        del sims
    return results if case["kind"] == "table" else results[0]
