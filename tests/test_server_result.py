"""Server.result without a GPU: the library and torch are stand-ins that record what they are asked for."""
import ctypes
import types

import pytest

from paper_2112_10034_gb300 import cox as c


class FakeTorch:
    """torch with two GPUs, of which `current` is current; default streams have the handle 0 everywhere."""
    float32, int32 = "float32", "int32"

    def __init__(self, current):
        self.cuda = types.SimpleNamespace(current_device=lambda: self.current, current_stream=self._stream)
        self.current = current
        self.outs, self.streams = [], []

    def _index(self, dev):
        if dev is None or dev == "cuda":
            return self.current
        return dev.index if hasattr(dev, "index") else int(dev)

    def device(self, kind, index):
        return types.SimpleNamespace(index=index)

    def _stream(self, dev=None):
        self.streams.append(self._index(dev))
        return types.SimpleNamespace(cuda_stream=0)

    def empty(self, n, dtype, device):
        self.outs.append((int(n), dtype, self._index(device)))
        return types.SimpleNamespace(data_ptr=lambda: 4096)


class FakeLib:
    """A done request of `count` elements; records the words read."""

    def __init__(self, count):
        self.count, self.words = count, []

    def cox_server_create(self, budget, max_requests, out):
        return c.COX_OK

    def cox_server_result(self, handle, ticket, out, count):
        ctypes.cast(count, ctypes.POINTER(ctypes.c_int64))[0] = self.count
        return c.COX_OK

    def cox_server_read(self, handle, ticket, dst, words, stream):
        self.words.append(words)
        return c.COX_OK

    def cox_server_destroy(self, handle):
        pass


def _server(monkeypatch, torch, lib):
    monkeypatch.setattr(c, "_torch", lambda: torch)
    monkeypatch.setattr(c, "lib", lambda: lib)
    return c.Server(1 << 20)


@pytest.mark.parametrize("kind", [c.COX_REQ_REDUCE, c.COX_REQ_SCAN, c.COX_REQ_COMPACT])
def test_the_copy_is_ordered_on_the_device_that_holds_it(kind, monkeypatch):
    """Another device than the server's is current.  The stream's handle says nothing of its
    device (0 is every device's default stream): the call goes to the current
    device's, so the output has to live there."""
    torch, lib = FakeTorch(current=0), FakeLib(7)
    srv = _server(monkeypatch, torch, lib)
    torch.current = 1
    srv.result(1, c.cox_request(kind, c.COX_I32, 32, 0, 7, 0, 16))
    assert [o[2] for o in torch.outs] == [1]
    assert torch.streams == [1]


@pytest.mark.parametrize("kind", [c.COX_REQ_SCAN, c.COX_REQ_COMPACT])
def test_the_length_is_the_servers(kind, monkeypatch):
    """A program may fill one request structure anew for each submission: it no
    longer describes the request whose result is read."""
    torch, lib = FakeTorch(current=0), FakeLib(7)
    srv = _server(monkeypatch, torch, lib)
    req = c.cox_request(kind, c.COX_I32, 32, 0, 7, 0, 16)
    req.n = 3
    srv.result(1, req)
    assert lib.words == [7] and torch.outs[0][0] == 7
