"""Calls of the one-call functions on several streams share a cached plan and its
workspace: they take turns.  The order of waits on the CPU with a fake device; results
on the GPU (needs a GB300)."""

import contextlib
import threading

import pytest

from paper_2110_01172_gb300 import binding, inputs

torch = pytest.importorskip("torch")


class Device:
    """A fake device: logs calls and waits as (what, stream); streams are ints."""

    def __init__(self, workspace):
        self.log, self.current, self.capturing, self.workspace = [], 1, set(), workspace

    def patch(self, monkeypatch):
        dev = self

        class Stream:
            def __init__(self, handle):
                self.cuda_stream = handle
                self.stream_id = handle if handle >= 100 else 7  # from 100 on: not PyTorch's own

            def wait_event(self, event):
                dev.log.append(("wait", self.cuda_stream, event.after))

        class Event:
            after = None

            def record(self):
                assert dev.current not in dev.capturing
                self.after = dev.current
                dev.log.append(("record", dev.current))

        class Plan:
            device, workspace_bytes = torch.device("cuda", 0), dev.workspace

            _h = None

            def __init__(self, *args):
                self._lib = self

            def _prep(self, x, out):
                return x, x

            def gbdct_exec_forward(self, *args):
                dev.log.append(("call", dev.current))
                return binding.OK

            def forward(self, x, out=None):
                self.gbdct_exec_forward()
                return x

        @contextlib.contextmanager
        def on(stream):
            was, dev.current = dev.current, stream.cuda_stream
            yield
            dev.current = was

        monkeypatch.setattr(binding, "Plan", Plan)
        monkeypatch.setattr(binding, "_plans", {})
        monkeypatch.setattr(binding, "_current_stream", lambda index: dev.current)
        for name, value in {"device": lambda d: contextlib.nullcontext(), "stream": on, "Event": Event,
                            "current_stream": lambda d=None: Stream(dev.current),
                            "is_current_stream_capturing": lambda: dev.current in dev.capturing}.items():
            monkeypatch.setattr(torch.cuda, name, value)

    def call(self, stream):
        self.current = stream
        binding.dct2(torch.zeros(4, 4))


def test_a_stream_waits_for_the_last_one(monkeypatch):
    dev = Device(workspace=64)
    dev.patch(monkeypatch)
    for s in (1, 1, 2, 2, 1):
        dev.call(s)
    assert dev.log == [("call", 1), ("call", 1), ("record", 1), ("wait", 2, 1), ("call", 2), ("call", 2),
                       ("record", 2), ("wait", 1, 2), ("call", 1)]


def test_no_order_without_a_workspace(monkeypatch):
    dev = Device(workspace=0)
    dev.patch(monkeypatch)
    for s in (1, 2, 1):
        dev.call(s)
    assert dev.log == [("call", 1), ("call", 2), ("call", 1)]


def test_streams_that_may_be_gone_and_captures(monkeypatch):
    dev = Device(workspace=64)
    dev.patch(monkeypatch)
    for s in (100, 1):  # the event of a stream that PyTorch does not own is recorded while it exists
        dev.call(s)
    assert dev.log == [("call", 100), ("record", 100), ("wait", 1, 100), ("call", 1)]
    dev.log.clear()
    dev.capturing = {3}
    for s in (3, 1, 2):  # a captured call neither waits nor counts as the last one
        dev.call(s)
    assert dev.log == [("call", 3), ("call", 1), ("record", 1), ("wait", 2, 1), ("call", 2)]
    dev.log.clear()
    dev.capturing = {2}
    dev.call(1)  # nothing can be recorded on a stream that another thread captures
    assert dev.log == [("call", 1)]


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(1024, 1024), (64, 512), (16, 256, 256)])
def test_results_on_two_streams_and_threads(shape):
    from paper_2110_01172_gb300 import dct2, dct3, idct2, idct3
    fwd, inv = (dct3, idct3) if len(shape) == 3 else (dct2, idct2)
    xs = [torch.rand(shape, generator=torch.Generator(device="cuda").manual_seed(i), device="cuda") for i in range(4)]
    ref = [fwd(x) for x in xs]
    back = [inv(r) for r in ref]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    got = {}

    def work(k, rounds):
        with torch.cuda.stream(streams[k % 2]):
            for r in range(rounds):
                y = fwd(xs[k])
                got[k, r] = (y, inv(y))

    for r in range(8):  # alternating from one thread
        for k in range(4):
            work(k, 1)
        torch.cuda.synchronize()
        assert all(torch.equal(got[k, 0][0], ref[k]) and torch.equal(got[k, 0][1], back[k]) for k in range(4))
    threads = [threading.Thread(target=work, args=(k, 20)) for k in range(4)]
    [t.start() for t in threads]
    [t.join() for t in threads]
    torch.cuda.synchronize()
    assert len(got) >= 80
    assert all(torch.equal(y, ref[k]) and torch.equal(z, back[k]) for (k, _), (y, z) in got.items())


@pytest.mark.gpu
def test_captured_call_replays():
    from paper_2110_01172_gb300 import dct2
    x = torch.from_numpy(inputs.uniform((256, 256), seed=5)).cuda()
    ref = dct2(x).clone()
    out, g = torch.zeros_like(x), torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        dct2(x, out)
    g.replay()
    assert torch.equal(out, ref) and torch.equal(dct2(x), ref)
