"""The binding's kept workspaces, on the CPU with a stand-in for the C entry
point: a workspace is created, and grown, on the stream that the call runs on,
so that its zero-fill comes before the call's kernels and its memory is given
back in that stream's order."""
import contextlib

import torch

import paper_2606_00535_gb300 as dreams


class Stream:
    def __init__(self, handle, device):
        self.cuda_stream, self.device = handle, device


def test_kept_workspace_belongs_to_the_calls_stream(monkeypatch):
    dev = torch.device("cuda", 0)
    current, made = [None], []
    need = 512

    @contextlib.contextmanager
    def use(stream):
        before, current[0] = current[0], stream if stream is not None else current[0]
        yield
        current[0] = before

    class Memory:
        def __init__(self, n):
            self.n = n
            made.append((n, current[0]))

        def data_ptr(self):
            return 4096

        def numel(self):
            return self.n

    def entry(name, device, args):
        return dreams.ERR_WORKSPACE if args[1] < need else dreams.OK

    monkeypatch.setattr(dreams, "_WS", {})
    monkeypatch.setattr(dreams, "_status_of", entry)
    monkeypatch.setattr(torch.cuda, "stream", use)
    monkeypatch.setattr(torch, "zeros", lambda n, dtype, device: Memory(n))
    side = Stream(77, dev)
    for need in (512, 256, 1024):
        dreams._call_ws("entry", dev, "kind", lambda: need, None, side, ())
    assert made == [(512, side), (1024, side)]
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda index: 5, raising=False)
    dreams._call_ws("entry", dev, "kind", lambda: need, None, None, ())
    assert made[2:] == [(1024, None)]  # no stream given: the current one
