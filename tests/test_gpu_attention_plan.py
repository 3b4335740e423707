"""Decode attention's plan: the prefix sum in every CTA's shared memory up to 4096 sequences, in a kernel of its own
beyond, against the oracle (the tolerance of every attention test); empty sequences among the others."""
import numpy as np
import pytest
import torch

import oracle
import workloads as W
from helpers import case_to_dev, dev, float_close, umim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 383, 384, 385, 4096, 4097])
def test_many_sequences_match_oracle(B):
    m = umim()
    lens = np.random.default_rng(B).integers(0, 40, size=B)
    lens[0], lens[-1] = 0 if B > 1 else 5, 17
    c = W.decode_case(50 + B, lens=lens, n_q_heads=2, n_kv_heads=1, head_dim=64, n_spans=[0] * B)
    g = case_to_dev(c, dev())
    status = m.new_status(dev())
    out = m.umim_decode_attention(g["q"], g["pool"], 0, g["bt"], g["lens"], dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = oracle.decode_attention(W.bits(c.q), W.bits(c.pool), 0, c.block_table.numpy(), c.seq_lens.numpy())
    float_close(out.cpu().double().numpy(), ref)
