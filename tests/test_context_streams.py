"""Contexts that follow torch's current stream (the ones that the autograd functions and sasa() keep for
every stream and thread): their calls share one scratch, so calls on different streams are put in order,
and two threads' calls come one after the other.  On the CPU with stand-ins for the library and torch's
streams; on a GPU with two streams."""
import threading
import time
import types

import numpy as np
import pytest


class _Stream:
    def __init__(self, handle, stream_id=None, capturing=False):
        self.cuda_stream, self.capturing = handle, capturing
        self.stream_id = handle if stream_id is None else stream_id
        self.waited = []

    def wait_stream(self, other):
        self.waited.append(other.cuda_stream)


class _Fake:
    """The library and torch.cuda as far as a call needs them; current is one stream per thread."""

    def __init__(self, monkeypatch):
        import torch
        from paper_2401_10462_gb300 import api
        self.tls, self.bound, self.calls, self.inside, self.overlap = threading.local(), [], [], 0, False
        me = self

        class On:
            def __init__(self, s):
                self.s = s

            def __enter__(self):
                self.old, me.tls.cur = me.tls.cur, self.s

            def __exit__(self, *a):
                me.tls.cur = self.old

        def call(*a):
            me.inside += 1
            me.overlap |= me.inside > 1
            me.calls.append((me.bound[-1], me.tls.cur.cuda_stream))
            time.sleep(0.002)
            me.inside -= 1
            return 0

        lib = types.SimpleNamespace(
            dsasa_default_config=lambda *a: None, dsasa_create=lambda *a: 0, dsasa_destroy=lambda *a: None,
            dsasa_set_stream=lambda h, s: self.bound.append(s.value or 0), dsasa_compute_vjp=call)
        monkeypatch.setattr(api, "_lib", lib)
        monkeypatch.setattr(api, "_check_tensor", lambda *a: None)
        monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: self.tls.cur)
        monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: self.tls.cur.capturing)
        monkeypatch.setattr(torch.cuda, "stream", On)
        self.tls.cur = _Stream(0)
        self.ctx = api.Context()

    def run(self, stream):
        self.tls.cur = stream
        self.ctx.compute(np.zeros((1, 3)), np.ones(1), np.zeros(1))


def test_calls_on_other_streams_wait(monkeypatch):
    f = _Fake(monkeypatch)
    a, b, default = _Stream(0x1000, 3), _Stream(0x2000, 5), _Stream(0)
    for s in (default, default, a, a, b, default):
        f.run(s)
    assert all(bound == cur for bound, cur in f.calls)        # the library enqueues where torch is
    assert a.waited == [0] and b.waited == [0x1000] and default.waited == [0x2000]


def test_captured_and_foreign_streams(monkeypatch):
    """A captured call waits for nothing outside its graph, and the call after it for the last one that
    ran; a stream that torch does not own is not touched again."""
    f = _Fake(monkeypatch)
    a, cap, foreign, b = _Stream(0x1000, 3), _Stream(0x2000, 5, capturing=True), _Stream(0x3000), _Stream(0x4000, 7)
    f.run(a)
    f.run(cap)
    assert cap.waited == []
    cap.capturing = False
    f.run(cap)                       # the same stream, no longer capturing
    assert cap.waited == [0x1000]
    a.capturing = True               # (another thread captures there)
    f.run(b)
    assert b.waited == [0x2000]
    f.run(foreign)
    f.run(b)
    assert foreign.waited == [0x4000] and b.waited == [0x2000]
    assert all(bound == cur for bound, cur in f.calls)


def test_threads_take_turns(monkeypatch):
    f = _Fake(monkeypatch)
    streams = [_Stream(0x1000, 3), _Stream(0x2000, 5)]

    def work(s):
        for _ in range(20):
            f.run(s)
    ts = [threading.Thread(target=work, args=(s,)) for s in streams]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not f.overlap and len(f.calls) == 40 and all(bound == cur for bound, cur in f.calls)


@pytest.mark.gpu
def test_autograd_on_two_streams(gen):
    """Energies of two molecules on two streams at once through the shared context: each equals the
    result of a call alone, bit by bit."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_10462_gb300 import autograd as ag
    mols = [gen.globule(6000, 1), gen.rna(2500, 2)]
    dev = [(torch.as_tensor(m.coords, device="cuda"), torch.as_tensor(m.radii, device="cuda")) for m in mols]

    def one(k):
        x = dev[k][0].clone().requires_grad_(True)
        e, areas = ag.nonpolar_energy(x, dev[k][1])
        (g,) = torch.autograd.grad(e, x)
        return areas.detach(), g
    ref = [one(0), one(1)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for s in streams:
        s.wait_stream(torch.cuda.current_stream())
    got = []
    for _ in range(10):
        for k, s in enumerate(streams):
            with torch.cuda.stream(s):
                got.append((k, one(k)))
    torch.cuda.synchronize()
    for k, (a, g) in got:
        assert torch.equal(a, ref[k][0]) and torch.equal(g, ref[k][1])
