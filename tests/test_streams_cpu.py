"""Calls with an explicit stream, on the CPU: the stream calls and the C functions
are fakes, and every buffer that a call allocates has to be allocated while its
stream is the current one (the pool the caching allocator takes it from)."""
import contextlib
import types

import pytest
import torch

from paper_2509_24416_gb300 import clq

HERE, SIDE = 3, 7
K, N, M, b = 128, 8, 4, 32


class FakeStream:
    def __init__(self, handle, log):
        self.cuda_stream, self.log = handle, log

    def wait_stream(self, other):
        self.log.append(("wait", self.cuda_stream, other.cuda_stream))


@pytest.fixture
def fake(monkeypatch):
    f = types.SimpleNamespace(current=HERE, log=[])

    @contextlib.contextmanager
    def stream(s):
        before, f.current = f.current, s.cuda_stream
        yield
        f.current = before

    f.side = FakeStream(SIDE, f.log)
    monkeypatch.setattr(torch.cuda, "stream", stream)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: FakeStream(f.current, f.log))
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "ExternalStream", lambda h: FakeStream(h, f.log))
    monkeypatch.setattr(clq, "_raw_stream", lambda device: f.current)
    empty = torch.empty

    def logged(*a, **k):
        f.log.append(("empty", f.current))
        return empty(*a, **k).zero_()

    monkeypatch.setattr(torch, "empty", logged)
    for name in clq.EXPORTS:
        if hasattr(clq, name):  # the stream is the last argument of those called here
            monkeypatch.setattr(clq, name, lambda *a, name=name: f.log.append((name, a[-1])) or 0)
    monkeypatch.setattr(clq, "clq_clip_search_workspace_size", lambda *a: 256)
    monkeypatch.setattr(clq, "clq_fused_linear_workspace_size", lambda *a: 256)
    monkeypatch.setattr(clq, "_host", types.SimpleNamespace(
        layer=lambda *a: f.log.append(("native", f.current)) or torch.zeros(M, N)))
    return f


X = torch.zeros(M, K, dtype=torch.float16)
W = torch.zeros(N, K, dtype=torch.float16)
PERM = torch.arange(K, dtype=torch.int32)
Q, S = torch.zeros(M, K, dtype=torch.uint8), torch.zeros(M)
WE, SW = torch.zeros(N, K, dtype=torch.uint8), torch.zeros(N)


def _layer():
    return clq.PreparedLinear(None, SW, PERM, b, We=WE)


def test_host_pipeline_buffers(fake, monkeypatch):
    made, recorded = [], []
    monkeypatch.setattr(torch.cuda, "Event", lambda *a, **k: None)
    monkeypatch.setattr(torch.cuda, "Stream", lambda device: made.append(
        FakeStream(20 + len(made), fake.log)) or made[-1])
    monkeypatch.setattr(clq, "_record", lambda ts, s: recorded.extend(
        (t.data_ptr(), s.cuda_stream) for t in ts if t is not None), raising=False)
    p = clq.HostPipeline([(_layer(), M, K, N)], torch.float16, "cpu", fused=True)
    # behind the current stream's work on the blocks the buffers are made of
    last = max(i for i, e in enumerate(fake.log) if e[0] == "empty")
    assert {("wait", s.cuda_stream, HERE) for s in made} <= set(fake.log[last + 1:])
    assert len(made) == 3
    # and the blocks go back only behind the streams that use them
    want = [(t, s) for t in p.xd for s in (p.s_in, p.s_comp)]
    want += [(t, s) for t in p.yd for s in (p.s_comp, p.s_out)]
    want += [(t, p.s_comp) for t in p.xq + p.sx + p.ws]
    assert {(t.data_ptr(), s.cuda_stream) for t, s in want} <= set(recorded)


CALLS = {
    "outlier_scores": lambda s: clq.outlier_scores(X[None], stream=s),
    "outlier_scores_range": lambda s: clq.outlier_scores(X[None], "range", s),
    "build_permutation_device": lambda s: clq.build_permutation_device(torch.zeros(K), s),
    "prepare_weights": lambda s: clq.prepare_weights(W, PERM, b, with_rot=True, stream=s),
    "rotate_quant_act": lambda s: clq.rotate_quant_act(X, PERM, b, clq.CLQ_CODES_E4M3, None, None,
                                                       True, s),
    "rotate_quant_act_asym": lambda s: clq.rotate_quant_act_asym(X, PERM, b, stream=s),
    "weight_code_sums": lambda s: clq.weight_code_sums(WE, K, s),
    "expand_weights": lambda s: clq.expand_weights(WE[:, :K // 2], s),
    "convert_codes": lambda s: clq.convert_codes(WE, K, clq.CLQ_CODES_INT4_PACKED, stream=s),
    "w4a4_linear": lambda s: clq.w4a4_linear(Q, S, WE, SW, b, K, stream=s),
    "linear": lambda s: clq.linear(Q, S, WE, SW, b, K, with_acc=True, stream=s),
    "linear_asym": lambda s: clq.linear_asym(Q, S, S, WE, SW, SW, b, K, stream=s),
    "clip_search": lambda s: clq.clip_search(W, PERM, b, X, torch.zeros(M, N), stream=s),
    "fused_linear": lambda s: clq.fused_linear(X, PERM, b, WE, SW, stream=s),
    "layer": lambda s: _layer()(X, stream=s),
    "layer_buffer": lambda s: _layer()(X, stream=s, Y=torch.zeros(M, N, dtype=torch.float16)),
    "layer_fused": lambda s: _layer()(X, fused=True, stream=s),
    "calibrate": lambda s: clq.PreparedLinear.calibrate(W, X[None], b, stream=s),
    "calibrate_clip": lambda s: clq.PreparedLinear.calibrate(W, X[None], b, stream=s,
                                                             clip_grid=(0.0, 0.01)),
}


def test_only_new_results_are_recorded(fake, monkeypatch):
    recorded = []
    monkeypatch.setattr(clq, "_record", lambda ts, s: recorded.extend((t, s.cuda_stream)
                                                                      for t in ts))
    Y = torch.zeros(M, N, dtype=torch.float16)
    out, acc = clq.linear(Q, S, WE, SW, b, K, Y=Y, with_acc=True, stream=fake.side)
    assert out is Y and len(recorded) == 1
    assert recorded[0][0] is acc and recorded[0][1] == HERE
    assert _layer()(X, stream=fake.side, Y=Y) is Y and len(recorded) == 1


@pytest.mark.parametrize("name", sorted(CALLS))
def test_buffers_belong_to_the_calls_stream(fake, name):
    CALLS[name](fake.side)
    work = [e for e in fake.log if e[0] != "wait"]
    assert work and all(e[-1] == SIDE for e in work), fake.log
    if name.startswith("calibrate"):  # behind the caller's work, in front of its next
        assert fake.log[0] == ("wait", SIDE, HERE) and fake.log[-1] == ("wait", HERE, SIDE)
    assert fake.current == HERE
    # without a stream, or with the current one: the current stream
    for s in (None, FakeStream(HERE, fake.log)):
        fake.log.clear()
        CALLS[name](s)
        assert fake.log and all(e[-1] == HERE for e in fake.log), fake.log
