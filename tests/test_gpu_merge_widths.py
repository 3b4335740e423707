"""The merge module with heads wider than 1024 columns (pooled by a CTA per span) at widths that do not fill a whole
number of column chunks per thread, against the float64 oracle (the tolerance of every merge test)."""
import pytest
import torch

import oracle
from oracle import merge as M
import workloads as W
from helpers import dev, float_close, umim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,h", [(1536, 1), (2560, 1), (3072, 2), (3584, 1), (5120, 4), (5632, 2), (6144, 1), (8192, 4)])
def test_wide_heads_match_oracle(d, h):
    m, on = umim(), dev()
    c = W.merge_case(760 + d, vocab=300, d=d, h=h, n_spans=11, kmin=1, kmax=4)
    status = m.new_status(on)
    z = m.umim_merge_spans(c.table.to(on), c.token_ids.to(on), c.span_offsets.to(on), c.weights.to(on), dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    wf = M.weights_f64({n: W.bits(v) for n, v in c.weights.tensors().items()})
    float_close(z.cpu().double().numpy(),
                oracle.merge_spans(W.bits(c.table), c.token_ids.numpy(), c.span_offsets.numpy(), wf, h))
