"""Prefill attention by the kernel that takes one head at a time (odd groups at every size), with many units a CTA: at
least five, of several query tiles' keys each, so that its rings, barriers and the four records of units in flight
are all used again; every row against the oracle within the tolerance of every prefill test."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from helpers import dev, float_close, umim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,hq,hkv,d", [(710, 28, 4, 128), (711, 8, 8, 64), (712, 9, 3, 64), (713, 7, 1, 128)])
def test_many_units_a_cta_match_oracle(seed, hq, hkv, d):
    m, dv = umim(), dev()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert hq // hkv % 2 == 1   # odd: the one-head kernel, two CTAs an SM
    r = np.random.default_rng(seed)
    lens = [1000, 129, 0, 640, 1]
    while sum(-(-n // 128) for n in lens) * hq < 10 * sms:
        lens.append(int(r.integers(200, 700)))
    r.shuffle(lens)
    T = sum(lens)
    # V of a quarter: the output's bf16 rounding stays below the absolute tolerance (as in the edge tests)
    q, k, v = (W.bf16_normal((T, h, d), std, seed * 10 + i, dv)
               for i, (h, std) in enumerate(((hq, 1.0), (hkv, 1.0), (hkv, 0.25))))
    cu = torch.tensor(np.concatenate([[0], np.cumsum(lens)]), dtype=torch.int32, device=dv)
    status = m.new_status(dv)
    out = m.umim_prefill_attention(q, k, v, cu, dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    float_close(out.cpu().double().numpy(), oracle.prefill_attention(W.bits(q), W.bits(k), W.bits(v), cu.cpu().numpy()))
