"""The order that the autograd wrappers give calls on a kept context, with stand-ins for the
library, the streams and the tensors: each call's stream waits for the event that the call
before recorded, before the context is bound again, whichever stream it ran on."""
import types

import pytest

torch = pytest.importorskip("torch")


class _Stream:
    def __init__(self, log, handle):
        self.log, self.cuda_stream = log, handle

    def __eq__(self, other):
        return self.cuda_stream == other.cuda_stream

    def wait_event(self, event):
        self.log.append(("wait", event.recorded))


class _Tensor:
    dtype = torch.float32
    device = types.SimpleNamespace(index=0)

    def __init__(self, *shape):
        self.shape = shape

    def record_stream(self, stream):
        pass


@pytest.mark.parametrize("handles", [(1, 1, 1), (1, 2, 1), (2, 2, 1)])
def test_a_call_waits_for_the_one_before(monkeypatch, handles):
    from paper_1301_3389_gb300 import autograd
    log = []

    class Event:
        recorded = None

        def record(self, stream):
            self.recorded = len(log)

    lib = types.SimpleNamespace(
        DNA_F64=0, DNA_F32=1, make_opts=lambda **k: None, dna_create=lambda *a: 7,
        dna_destroy=lambda c: None, dna_set_stream=lambda c, s: None,
        dna_bind=lambda c, V, W, H: log.append(("bind", c)))
    streams = iter([_Stream(log, h) for h in handles])
    monkeypatch.setattr(autograd, "L", lib)
    monkeypatch.setattr(autograd, "_local", types.SimpleNamespace())
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: next(streams))
    monkeypatch.setattr(torch.cuda, "Event", Event)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    V, W, H = _Tensor(5, 6), _Tensor(5, 2), _Tensor(2, 6)
    ends = []
    for _ in handles:
        with autograd._Ctx(V, W, H):
            log.append(("call",))
        ends.append(len(log))
    assert log == [("bind", 7), ("call",),
                   ("wait", ends[0]), ("bind", 7), ("call",),
                   ("wait", ends[1]), ("bind", 7), ("call",)]
