"""Prefill attention over enough units for two heads at a time, against the oracle within the tolerance of every
prefill test: sequences of every length about the edges of the 128-row tiles, the 128-key tiles and their halves,
empty ones, several tiles long ones, more units than CTAs; the smallest even group, the largest, both head dims."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from helpers import dev, float_close, umim

pytestmark = pytest.mark.gpu

EDGES = [1, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129, 0, 191, 192, 193, 255, 256, 257, 321, 17]


@pytest.mark.parametrize("lens,hq,hkv,d", [
    (EDGES * 2, 32, 8, 128), (EDGES * 3, 16, 8, 64), (EDGES * 2 + [900], 32, 2, 128), ([700] + EDGES * 2, 32, 16, 64),
    ([530] * 8, 32, 8, 64),
])
def test_pairs_of_heads_match_oracle(lens, hq, hkv, d):
    m, dv = umim(), dev()
    T = sum(lens) + 3
    # (as in the other edge test: V of a quarter, so that rows of one key stay below 4 and bf16's rounding of the
    # output, 2^-9 of it, below the absolute tolerance)
    q, k = (W.bf16_normal((T, h, d), 1.0, 700 + i, dv) for i, h in enumerate((hq, hkv)))
    v = W.bf16_normal((T, hkv, d), 0.25, 702, dv)
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32, device=dv)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert 2 * (T // 128 + len(lens)) * (hq // 2) >= 7 * sms   # the pair kernel's range
    out = torch.full_like(q, 7.0)
    status = m.new_status(dv)
    m.umim_prefill_attention(q, k, v, cu, out=out, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    want = oracle.prefill_attention(W.bits(q), W.bits(k), W.bits(v), cu.cpu().numpy())
    got = out.cpu().double().numpy()
    float_close(got[:T - 3], want[:T - 3], "prefill")
    assert np.all(got[T - 3:] == 7.0)
