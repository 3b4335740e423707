"""Calls captured once as a CUDA graph and replayed on other inputs in the same buffers, against the eager call bit for
bit: the products split over clusters with their early launches, the rollback's one plan-and-map kernel, both prefill
kernels with the plan in the V transpose, attention with the plan in its CTAs, the per-layer step's shared merge."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import case_to_dev, dev, umim

pytestmark = pytest.mark.gpu


def _merge(m, d, S):
    cases = [W.merge_case(850 + d + i, vocab=300, d=d, h=4, n_spans=S, kmin=2, kmax=2) for i in range(2)]
    w, offs = cases[0].weights.to(dev()), cases[0].span_offsets.to(dev())
    ws = m.workspace(m.umim_merge_spans_workspace_size(2 * S, S, d), dev())
    z = torch.empty(S, d, device=dev())
    inputs = [[c.table.to(dev()), c.token_ids.to(dev())] for c in cases]
    return inputs, [z], lambda t, ids: m.umim_merge_spans(t, ids, offs, w, surrogates=z, workspace_buf=ws)


def _rollback(m, lens):
    g = [case_to_dev(W.decode_case(860 + i, lens=lens, n_q_heads=4, n_kv_heads=2, head_dim=64, n_spans=[9] * len(lens)),
                     dev()) for i in range(2)]
    names = ("pool", "bt", "lens", "offs", "st", "ln", "sk", "sv")
    freed = torch.empty(g[0]["bt"].numel(), dtype=torch.int32, device=dev())
    ws = m.workspace(m.umim_kv_rollback_workspace_size(len(lens), g[0]["st"].numel(), g[0]["bt"].shape[1], 1, 2, 64), dev())
    freq = (1e4 ** (-torch.arange(32, device=dev()) / 32.0)).float()
    out = [torch.empty_like(g[0][n]) for n in ("pool", "bt", "lens")] + [freed]

    def call(*x):
        for o, t in zip(out[:3], x):
            o.copy_(t)
        freed.fill_(-1)
        m.umim_kv_rollback(out[0], out[1], out[2], *x[3:], freed_pages=freed, workspace_buf=ws, rope_inv_freq=freq)
    return [[c[n] for n in names] for c in g], out, call


def _prefill(m, lens, hq, hkv):
    T, dv = sum(lens), dev()
    cu = [torch.tensor(np.concatenate([[0], np.cumsum(x)]), dtype=torch.int32, device=dv) for x in (lens, lens[::-1])]
    inputs = [[W.bf16_normal((T, h, 64), 1.0, 870 + 3 * i + j, dv) for j, h in enumerate((hq, hkv, hkv))] + [cu[i]]
              for i in range(2)]
    out = torch.empty_like(inputs[0][0])
    ws = m.workspace(m.umim_prefill_attention_workspace_size(len(lens), T, hkv, 64), dv)
    return inputs, [out], lambda q, k, v, c: m.umim_prefill_attention(q, k, v, c, out=out, workspace_buf=ws)


def _attention(m, lens, step):
    g = [case_to_dev(W.decode_case(880 + i, lens=x, n_q_heads=8, n_kv_heads=2, head_dim=64, coverage=0.0), dev())
         for i, x in enumerate((lens, lens[::-1]))]
    pages = max(c["pool"].shape[1] for c in g)
    assert all(c["pool"].shape[1] == pages for c in g)
    out = torch.empty_like(g[0]["q"])
    inputs = [[c[n] for n in ("q", "pool", "bt", "lens")] for c in g]
    B = len(lens)
    if step:
        new = [W.bf16_normal((B, 2, 64), 1.0, 890 + i, dev()) for i in range(2)]
        ws = m.workspace(m.umim_decode_layer_step_workspace_size(B, 2, 64), dev())
        return [x + [n] for x, n in zip(inputs, new)], [out], lambda q, p, bt, l, n: m.umim_decode_layer_step(
            q, p, 0, bt, l, n, n, out=out, workspace_buf=ws)
    ws = m.workspace(m.umim_decode_attention_workspace_size(B, 8, 2, 64), dev())
    return inputs, [out], lambda q, p, bt, l: m.umim_decode_attention(q, p, 0, bt, l, out=out, workspace_buf=ws)


@pytest.mark.parametrize("make,args", [
    (_merge, (512, 9)), (_merge, (512, 1000)), (_merge, (1536, 300)), (_merge, (2048, 1100)),
    (_rollback, ([700, 33, 400],)), (_rollback, ([4200, 50],)),
    (_prefill, ([5, 129, 64, 300], 8, 2)), (_prefill, ([300] * 60, 8, 2)),
    (_attention, ([9001, 17, 333], False)), (_attention, ([9001, 17, 333], True)),
], ids=["merge8", "merge4", "merge2", "merge_whole", "plan_map", "long_table", "prefill", "prefill_pair", "attention",
        "layer_step"])
def test_replay_on_other_inputs_equals_the_eager_call(make, args):
    m = umim()
    (first, second), outs, call = make(m, *args)
    buffers = [t.clone() for t in first]
    want = []
    for x in (first, second):
        call(*x)
        torch.cuda.synchronize()
        want.append([o.clone() for o in outs])
    call(*buffers)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(*buffers)
    for x, w in ((second, want[1]), (first, want[0]), (second, want[1])):
        for b, t in zip(buffers, x):
            b.copy_(t)
        graph.replay()
        torch.cuda.synchronize()
        for o, v in zip(outs, w):
            assert torch.equal(o, v)
