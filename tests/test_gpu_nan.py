"""Scores of NaN and of -inf in a long sequence, wherever the split of the sequence puts them, against the oracle's
softmax: NaN makes the row NaN (pieces in which every score is NaN have no maximum, and no merge of pieces may take them
for empty ones), -inf weighs 0, and only -inf scores make it NaN again.  The other sequence stays as it is."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from helpers import dev, float_close, umim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["attention", "layer_step"])
@pytest.mark.parametrize("value", ["nan", "-inf"])
@pytest.mark.parametrize("lo,hi", [(0, 64), (3024, 4032), (4000, 9000), (5000, 5001), (9900, 12000), (0, 12000)])
@pytest.mark.parametrize("hq,d", [(5, 128), (16, 64)])
def test_scores_of_nan_and_minus_infinity(call, value, lo, hi, hq, d):
    m, dv = umim(), dev()
    lens = [12000, 300]
    c = W.decode_case(940 + d, lens=lens, n_q_heads=hq, n_kv_heads=1, head_dim=d, coverage=0.0, spare_pages=4,
                      extra_max_pages=1)
    t = np.arange(lo, hi)
    c.q[:, :, 0] = c.q[:, :, 0].abs() + 0.5   # the key's element below times this: the value itself, in every head
    c.pool[0, torch.from_numpy(c.block_table.numpy()[0, t // 16]).long(), 0, 0, torch.from_numpy(t % 16), 0] = float(value)
    pool, bt, sl, q = c.pool.to(dv), c.block_table.to(dv), c.seq_lens.to(dv), c.q.to(dv)
    status = m.new_status(dv)
    if call == "attention":
        out = m.umim_decode_attention(q, pool, 0, bt, sl, dev_status=status)
        want = oracle.decode_attention(W.bits(c.q), W.bits(c.pool), 0, c.block_table.numpy(), c.seq_lens.numpy())
    else:
        new = W.bf16_normal((2, 1, d), 1.0, 941, dv)
        pages = torch.tensor([p for p in range(c.n_pages) if p not in set(c.block_table.numpy().ravel().tolist())][:2],
                             dtype=torch.int32, device=dv)
        out = m.umim_decode_layer_step(q, pool, 0, bt, sl, new, new, new_pages=pages, commit=True, dev_status=status)
        torch.cuda.synchronize()
        want = oracle.decode_attention(W.bits(c.q), W.bits(pool), 0, bt.cpu().numpy(), sl.cpu().numpy())
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    got = out.cpu().double().numpy()
    if value == "nan" or (hi - lo == 12000 and call == "attention"):
        assert np.all(np.isnan(want[0])) and np.all(np.isnan(got[0]))
    else:
        float_close(got[0], want[0])
    float_close(got[1], want[1])


@pytest.mark.parametrize("value", ["nan", "-inf"])
@pytest.mark.parametrize("hq,hkv,d", [(32, 8, 128), (16, 8, 64), (7, 1, 128)])   # two heads at a time, and one
def test_prefill_scores_of_nan_and_minus_infinity(value, hq, hkv, d):
    """One key of the middle of a sequence, the last one of another: rows from it on are NaN, or weigh it 0; rows before
    it, the other heads' and the other sequences' rows (in the same tiles of keys) are untouched."""
    m, dv = umim(), dev()
    lens = [300, 70, 515, 129] + [260] * {32: 16, 16: 30, 7: 1}[hq]
    T, cu_np = sum(lens), np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert (hq // hkv % 2 == 0 and 2 * (T // 128 + len(lens)) * (hq // 2) >= 7 * sms) == (hq > 7)
    # (V of a quarter, as in the other edge tests: the output's rounding stays below the absolute tolerance)
    q, k, v = (W.bf16_normal((T, h, d), s, 950 + i, dv) for i, (h, s) in enumerate(((hq, 1.0), (hkv, 1.0), (hkv, 0.25))))
    q[:, :, 0] = q[:, :, 0].abs() + 0.5
    hit = [int(cu_np[2]) + 197, int(cu_np[2]) - 1]
    for t in hit:
        k[t, 0, 0] = float(value)
    status = m.new_status(dv)
    out = m.umim_prefill_attention(q, k, v, torch.from_numpy(cu_np).to(dv), dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    want = oracle.prefill_attention(W.bits(q), W.bits(k), W.bits(v), cu_np)
    got = out.cpu().double().numpy()
    nan = np.isnan(want)
    assert nan.any() == (value == "nan")
    np.testing.assert_array_equal(np.isnan(got), nan)
    float_close(np.where(nan, 0.0, got), np.where(nan, 0.0, want))
