"""Calls of different sizes from several host threads at once.  A kernel's limit of dynamic shared memory is one value per
device, and ctypes drops the interpreter's lock: a call that set it to its own size could find the limit of the other
thread's smaller call in force at its launch and fail."""
import threading

import pytest
import torch

import workloads as W
from helpers import case_to_dev, dev, umim

pytestmark = pytest.mark.gpu

ROUNDS = 5000   # calls a thread; of 5000 calls at the larger size about 150 failed


def _attention(m, B):
    g = case_to_dev(W.decode_case(810 + B, lens=[5] * B, n_q_heads=2, n_kv_heads=1, head_dim=64, n_spans=[0] * B), dev())
    out = torch.empty_like(g["q"])
    ws = m.workspace(m.umim_decode_attention_workspace_size(B, 2, 1, 64), dev())
    return lambda stream: m.umim_decode_attention(g["q"], g["pool"], 0, g["bt"], g["lens"], out=out, workspace_buf=ws,
                                                  stream=stream)


def _layer_step(m, B):
    g = case_to_dev(W.decode_case(820 + B, lens=[5] * B, n_q_heads=2, n_kv_heads=1, head_dim=64, n_spans=[0] * B), dev())
    new = torch.zeros(B, 1, 64, dtype=torch.bfloat16, device=dev())
    out = torch.empty_like(g["q"])
    ws = m.workspace(m.umim_decode_layer_step_workspace_size(B, 1, 64), dev())
    return lambda stream: m.umim_decode_layer_step(g["q"], g["pool"], 0, g["bt"], g["lens"], new, new, out=out,
                                                   workspace_buf=ws, stream=stream)


def _merge(m, dh):
    d = dh[0]
    c = W.merge_case(830 + d, vocab=50, d=d, h=dh[1], n_spans=3)
    table, ids, offs, w = (x.to(dev()) for x in (c.table, c.token_ids, c.span_offsets, c.weights))
    out = torch.empty(3, d, dtype=torch.float32, device=dev())
    ws = m.workspace(m.umim_merge_spans_workspace_size(ids.numel(), 3, d), dev())
    return lambda stream: m.umim_merge_spans(table, ids, offs, w, surrogates=out, workspace_buf=ws, stream=stream)


class _Recorder:
    """The library, noting the arguments of the call made through it."""

    def __init__(self, lib):
        self.lib = lib

    def __getattr__(self, name):
        fn = getattr(self.lib, name)

        def call(*args):
            self.call = fn, args
            return fn(*args)
        return call


@pytest.mark.parametrize("make,sizes", [
    (_attention, (1, 4096)), (_layer_step, (1, 4096)),
    (_merge, ((512, 4), (1024, 4))),    # pooling by a warp per head
    (_merge, ((1536, 1), (2048, 1))),   # by a CTA per span
], ids=["attention", "layer_step", "merge_heads", "merge_wide"])
def test_calls_of_two_sizes_from_four_threads(make, sizes, monkeypatch):
    m = umim()
    streams = [torch.cuda.Stream() for _ in range(4)]
    keep, calls = [], []
    rec = _Recorder(m.lib())
    for i, stream in enumerate(streams):   # two threads a size
        keep.append(make(m, sizes[i % 2]))
        torch.cuda.synchronize()
        with monkeypatch.context() as mp:
            mp.setattr(m, "lib", lambda: rec)
            keep[-1](stream)
        calls.append(rec.call)
    failed = [0] * len(calls)

    def loop(i):   # the recorded C call, so that nearly all of a thread's time is spent inside it
        fn, args = calls[i]
        for k in range(ROUNDS):
            failed[i] += fn(*args) != 0
            if k % 200 == 199:
                streams[i].synchronize()

    threads = [threading.Thread(target=loop, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert failed == [0] * len(calls)
