"""The merge module's products with K split over a cluster, at the edges of the 128-row tiles, against the float64
oracle (the tolerance of every merge test).  The splits named below are those of 152 SMs; that a size takes the split it
should is checked in test_gpu_merge_paths.py."""
import pytest
import torch

import oracle
from oracle import merge as M
import workloads as W
from helpers import dev, float_close, umim

pytestmark = pytest.mark.gpu


# at d = 512 (2 column tiles) on 152 SMs: 16 rows of tiles split 4 ways, 17 to 33 two ways, more not at all
@pytest.mark.parametrize("d,S,k", [
    (512, 1, 1), (512, 127, 1), (512, 128, 1), (512, 129, 1),   # both products split 8 ways
    (512, 300, 4),                                              # 4 and 8 ways
    (512, 700, 4),                                              # 2 and 8 ways
    (512, 1200, 4),                                             # whole tiles and 4 ways
    (512, 2100, 2),                                             # 2 and 2 ways, 33 and 17 rows of tiles
    (512, 4300, 1),                                             # whole tiles both
    (4096, 5, 3),                                               # 16 column tiles, 8 K steps a CTA
])
def test_split_products_match_oracle(d, S, k):
    m = umim()
    case = W.merge_case(700 + S, vocab=2000, d=d, h=4, n_spans=S, kmin=k, kmax=k)
    on = dev()
    status = m.new_status(on)
    z = m.umim_merge_spans(case.table.to(on), case.token_ids.to(on), case.span_offsets.to(on), case.weights.to(on),
                           dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    wf = M.weights_f64({n: W.bits(v) for n, v in case.weights.tensors().items()})
    float_close(z.cpu().double().numpy(),
                oracle.merge_spans(W.bits(case.table), case.token_ids.numpy(), case.span_offsets.numpy(), wf, 4))
