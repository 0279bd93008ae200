"""Host side of ``Layer.bind`` with a fake device: which device is current at its calls into the
library, what has completed when it returns, and what it asks about a stream under capture."""
import types

import numpy as np
import pytest
import torch

from paper_2003_06513_gb300 import _lib, api


class _Stream:
    def __init__(self, device, capturing=False):
        self.device, self.cuda_stream, self.capturing = device, 7 + device, capturing


class _FakeCuda:
    """Two devices; the calls in order, each with the device that was current."""

    def __init__(self, lib):
        self.lib, self.current, self.calls = lib, 0, []
        self.streams = [_Stream(0), _Stream(1)]
        self.now = self.streams[0]

    def _swap(self, device, stream):
        old = self.current, self.now
        self.current, self.now = device, stream
        return old

    def device(self, d):
        fake = self
        index = d.index if d.index is not None else fake.current

        class Guard:
            def __enter__(self):
                self.old = fake._swap(index, fake.streams[index])

            def __exit__(self, *a):
                fake.current, fake.now = self.old
        return Guard()

    def stream(self, s):
        fake = self

        class Guard:
            def __enter__(self):
                self.old = fake._swap(s.device, s)

            def __exit__(self, *a):
                fake.current, fake.now = self.old
        return Guard()

    def current_stream(self, device=None):
        return self.streams[device.index if device is not None and device.index is not None else self.current]

    def is_current_stream_capturing(self):
        return self.now.capturing

    # the library's calls
    def pp_bind_device(self, h, dev, n, stream):
        self.calls.append(("image", self.current, stream.value))
        return 0

    def pp_bind_tensor(self, h, dev, n, stream):
        self.calls.append(("tensor", self.current, stream.value))
        return 0

    def __getattr__(self, name):      # the rest of the library
        return getattr(self.lib, name)


@pytest.fixture
def fake(monkeypatch):
    f = _FakeCuda(_lib.load())
    f.capturing_synchronised = False

    def synchronize(s):
        assert not s.capturing, "a stream under capture was synchronised"
        f.calls.append(("done", f.current, s.cuda_stream))
    monkeypatch.setattr(_Stream, "synchronize", synchronize, raising=False)

    class Torch(types.ModuleType):
        cuda = f
        empty = staticmethod(lambda n, dtype, device: torch.empty(n, dtype=dtype))

        def __getattr__(self, name):
            return getattr(torch, name)
    monkeypatch.setattr(api, "torch", Torch("torch"))
    monkeypatch.setattr(_lib, "load", lambda *a, **k: f)
    return f


def _dense():
    return api.pp_pack(np.random.default_rng(0).standard_normal((16, 16, 3, 3)).astype(np.float32), None, 0.5)


def test_the_layers_device_is_current_at_every_call(fake):
    """The tensor-core weights are built by a kernel, which runs on the current device."""
    _dense().bind("cuda:1")
    assert [c[:2] for c in fake.calls if c[0] != "done"] == [("image", 1), ("tensor", 1)]
    assert fake.current == 0


def test_complete_on_return_whatever_the_layer_holds(fake):
    """Depthwise layers and weights of extreme range have no tensor-core weights; their image is copied
    all the same, and calls on any stream may follow."""
    w = np.random.default_rng(0).standard_normal((16, 1, 3, 3)).astype(np.float32)
    for layer, builds in ((_dense(), True), (api.pp_pack(w, None, 1.0, 16), False),
                          (api.pp_pack(np.full((8, 16, 3, 3), 1e-20, np.float32), None, 1.0), False)):
        fake.calls.clear()
        layer.bind("cuda")
        assert [c[0] for c in fake.calls] == ["image"] + ["tensor"] * builds + ["done"]


@pytest.mark.parametrize("capturing", ["given", "current"])
def test_a_stream_under_capture_is_not_synchronised(fake, capturing):
    """What counts is the stream that the work goes to, current or not."""
    side = _Stream(0, capturing=capturing == "given")
    fake.streams[0].capturing = capturing == "current"
    _dense().bind("cuda", stream=side)
    assert [c[2] for c in fake.calls] == [side.cuda_stream] * (2 if capturing == "given" else 3)
