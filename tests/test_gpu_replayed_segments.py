"""The parts of a step that are replayed as recorded graphs from their second use on give the bits of the first use."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
from paper_2010_04116_b200 import Model  # noqa: E402

pytestmark = pytest.mark.gpu


def _model(rng, K=3, n=2, Lh=0, **kw):
    m = Model(K, 1, 128, 4, 512, 300, n, 4, 48, head_layers=Lh, attn_bwd="two_kernels", **kw)
    for name in m.names:
        m.set_param(name, (rng.standard_normal(m.shapes[name]) * 0.05 + (1.0 if name.endswith(".g") else 0.0)).astype(np.float32))
    return m


def _batch(rng, B, T):
    return tuple(rng.integers(0, 300, size=(B, T)).astype(np.int32) for _ in range(2))


def _result(m, batch):
    m.train_step(*batch)
    losses = m.get_losses()
    m.sync()
    # weight matrices: sums of fixed order (vectors are summed atomically)
    return [losses] + [m.get_grad(name) for name in m.names if len(m.shapes[name]) == 2]


@pytest.mark.parametrize("kw", [{}, {"Lh": 1}, {"head_mode": "recompute"}, {"n": 1}])
def test_replay_equals_first_use_for_each_shape(kw):
    rng = np.random.default_rng(3)
    m = _model(rng, **kw)
    shapes = [(4, 48), (1, 48), (3, 31), (2, 1), (4, 17), (1, 7)]       # more than one stream's recordings hold
    batches = [_batch(rng, *s) for s in shapes]
    first = [_result(m, b) for b in batches]
    l0 = m.stats()[1]
    _result(m, batches[0])
    per_step = m.stats()[1] - l0
    for _ in range(3):
        for f, b in zip(first, batches):
            for x, y in zip(f, _result(m, b)):
                assert np.array_equal(x, y)
    l0 = m.stats()[1]
    _result(m, batches[0])
    assert m.stats()[1] - l0 == per_step                  # a replayed kernel counts like an enqueued one


def test_replay_after_the_rule_and_window_change():
    rng = np.random.default_rng(4)
    m = _model(rng, K=4, n=1)
    b = _batch(rng, 4, 48)
    seen = {}
    for n, rule in [(1, "sum"), (3, "sum"), (3, "mean"), (2, "far"), (1, "sum"), (3, "mean")] * 2:
        m.set_n(n)
        m.set_rule(rule)
        for _ in range(3):
            r = _result(m, b)
            if (n, rule) in seen:
                for x, y in zip(seen[n, rule], r):
                    assert np.array_equal(x, y)
            seen.setdefault((n, rule), r)


def test_recompute_head_with_micro_batches_is_recorded():
    """Every pass of an update is recorded, the accumulating ones of the recomputing head too: a recording that had to be given up
    would have left the reason in the model's last error."""
    rng = np.random.default_rng(5)
    m = _model(rng, head_mode="recompute")
    parts = [_batch(rng, 4, 48) for _ in range(3)]
    first = None
    for _ in range(4):
        m.set_micro_batches(3)
        for b in parts:
            r = _result(m, b)
        first = first or r
        for x, y in zip(first, r):
            assert np.array_equal(x, y)
        assert m.L.il_last_error(m._h) == b""


@pytest.mark.parametrize("kw", [{"K": 2}, {"K": 1, "n": 1}, {"K": 3, "Lh": 1, "head_mode": "recompute"}])
@pytest.mark.parametrize("with_batch", [True, False])
def test_a_caller_captures_a_step(kw, with_batch):
    """A step whose streams the caller is capturing goes into the caller's graph, after steps outside of it and before others, with
    the batch's copy or without it (then the graph runs on whatever batch is set before it)."""
    rng = np.random.default_rng(6)
    m = _model(rng, **kw)
    batches = [tuple(torch.tensor(x, device="cuda") for x in _batch(rng, 4, 48)) for _ in range(2)]
    ref = [_result(m, b) for b in batches]
    weights = [name for name in m.names if len(m.shapes[name]) == 2]
    graph = torch.cuda.CUDAGraph()
    if not with_batch:
        m.set_batch(*batches[0])
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=m.streams[0]):
        for s in m.streams[1:]:
            s.wait_stream(m.streams[0])
        if with_batch:
            m.set_batch(*batches[0])
        for k in range(m.K):
            m.forward_component(k)
            m.aux_head_loss(k)
        m.backward_nwise()
        for s in m.streams[1:]:
            m.streams[0].wait_stream(s)
    for i in [0] if with_batch else [0, 1, 0]:
        if not with_batch:
            _result(m, batches[i])                        # (as a step; what follows runs on the same ids)
        list(m._blocks.values())[1].fill_(77)             # the gradients
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        for x, name in zip(ref[i][1:], weights):
            assert np.array_equal(x, m.get_grad(name)), name
    del graph
    for i in [0, 1, 1, 0]:
        for x, y in zip(ref[i], _result(m, batches[i])):
            assert np.array_equal(x, y)
    assert m.L.il_last_error(m._h) == b""


def test_other_work_on_the_model_s_streams_is_not_recorded():
    """Another thread's kernels on a stream that the model works on (two models may share one of torch's streams) run once each."""
    rng = np.random.default_rng(7)
    m = _model(rng)
    counters = torch.zeros(len(m.streams), device="cuda")
    torch.cuda.synchronize()
    issued, stop, failed = [0] * len(m.streams), threading.Event(), []

    def other():
        try:
            while not stop.is_set():
                for i, s in enumerate(m.streams):
                    with torch.cuda.stream(s):
                        counters[i].add_(1)
                    issued[i] += 1
        except Exception as e:
            failed.append(e)
    t = threading.Thread(target=other)
    t.start()
    try:
        for B in range(1, 5):
            for T in range(1, 13):
                b = _batch(rng, B, T)
                for _ in range(3):
                    _result(m, b)
    finally:
        stop.set()
        t.join()
    torch.cuda.synchronize()
    assert not failed
    assert counters.tolist() == issued


def test_more_shapes_than_recordings_are_not_recorded_over_and_over():
    """Batch shapes in random order, more of them than a component keeps recordings for: those it has stay in use, the others are
    enqueued directly, and nothing waits for the stream in the middle of a step."""
    rng = np.random.default_rng(8)
    m = _model(rng)
    batches = [_batch(rng, 4, T) for T in range(6, 48, 4)]
    for i in rng.permutation(np.arange(8 * len(batches)) % len(batches)):
        m.train_step(*batches[i])
        m.sync()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU, torch.profiler.ProfilerActivity.CUDA]) as prof:
        for i in rng.permutation(np.arange(4 * len(batches)) % len(batches)):
            m.train_step(*batches[i])
    calls = {e.key: e.count for e in prof.key_averages()}
    assert sum(n for name, n in calls.items() if "GraphLaunch" in name) > 0, calls
    assert not [name for name in calls if "GraphInstantiate" in name or "StreamSynchronize" in name], calls


def test_recordings_follow_a_program_to_other_shapes():
    """Recordings that nobody has used for 1024 calls on their stream make room."""
    rng = np.random.default_rng(9)
    m = _model(rng)
    for T in range(6, 48, 4):
        b = _batch(rng, 4, T)
        for _ in range(3):
            m.train_step(*b)
    b = _batch(rng, 4, 48)
    first = _result(m, b)
    for i in range(270):
        m.train_step(*b)
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU, torch.profiler.ProfilerActivity.CUDA]) as prof:
        m.train_step(*b)
    calls = {e.key: e.count for e in prof.key_averages()}
    assert sum(n for name, n in calls.items() if "GraphLaunch" in name) == 4 * m.K, calls
    for x, y in zip(first, _result(m, b)):
        assert np.array_equal(x, y)
