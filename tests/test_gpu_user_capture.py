"""A caller that captures the ctx stream (day loops launched one by one, GABM_CUDA_GRAPHS=0): a
captured forward leaves the eager ones right before and after it is replayed, and a table
is not exchanged inside a capture."""
import numpy as np
import pytest
import torch

from paper_2207_09714_gb300 import capi, synth

from helpers import ensure_built, model, to_dev

pytestmark = pytest.mark.gpu

T = 20


@pytest.fixture
def setting(monkeypatch):
    ensure_built()
    monkeypatch.setenv("GABM_CUDA_GRAPHS", "0")
    pop = synth.population_small(n=4000, seed=6)
    stream = torch.cuda.Stream()
    dev = to_dev(np.full((1, T), 2.6, np.float32), np.full((1, T), 0.02, np.float32),
                 synth.SUSCEPTIBILITY[None, :].astype(np.float32))
    torch.cuda.synchronize()

    def run(ctx, n_seed):
        with torch.cuda.stream(stream):
            capi.gabm_forward(ctx, T, *dev, [n_seed])
        stream.synchronize()
        return capi.gabm_get_state(ctx)

    def make():
        return capi.gabm_create([pop], model(seed=3), stream=stream)

    return make, run, dev, stream


def test_eager_forward_after_a_captured_one(setting):
    make, run, dev, stream = setting
    want = {k: run(make(), k) for k in (10, 25)}
    assert not np.array_equal(want[10], want[25])
    ctx = make()
    assert np.array_equal(run(ctx, 10), want[10])
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        capi.gabm_forward(ctx, T, *dev, [25])
    assert np.array_equal(run(ctx, 25), want[25])   # the captured one, of as many seeds, has not run
    assert np.array_equal(run(ctx, 10), want[10])
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(capi.gabm_get_state(ctx), want[25])
    assert np.array_equal(run(ctx, 10), want[10])   # nor do the seeds of the replay stay


def test_no_table_is_set_inside_a_capture(setting):
    make, run, dev, stream = setting
    ctx = make()
    want = run(ctx, 10)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        D = dev[0] + 1.0
        with pytest.raises(capi.GabmError):
            capi.gabm_set_infectiousness(ctx, synth.infectiousness_table(T_E=0.2, T_I=1.3))
    assert np.array_equal(run(ctx, 10), want)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(D, dev[0] + 1.0)


def test_seeds_and_tables_of_forwards_still_queued(setting):
    """Calls that return before the stream has reached them keep the values they were given."""
    make, run, dev, stream = setting
    tables = [synth.infectiousness_table(T_E=e, T_I=1.3) for e in (0.2, 0.9)]
    want = []
    for k, c in enumerate(tables):
        ctx = make()
        capi.gabm_set_infectiousness(ctx, c)
        want.append(run(ctx, 10 + k))
    ctx = make()
    with torch.cuda.stream(stream):
        busy = torch.rand((4096, 4096), device="cuda")
        got = []
        for _ in range(8):
            for k, c in enumerate(tables):
                for _ in range(4):
                    busy = busy @ busy / 2048.0
                capi.gabm_set_infectiousness(ctx, c)
                capi.gabm_forward(ctx, T, *dev, [10 + k])
                got.append(capi.gabm_get_state(ctx, device=True))
    stream.synchronize()
    for i, e in enumerate(got):
        assert np.array_equal(e.cpu().numpy(), want[i % 2])
