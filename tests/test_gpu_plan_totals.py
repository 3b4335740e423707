"""The plan's prefix sums over the sequences, by one warp (four sequences a lane) up to 128 and by a block beyond:
rollbacks and prompt compactions of that many sequences, some without spans, bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import case_to_dev, compare_rollback, dev, oracle_rollback, umim
from test_gpu_compaction import test_compaction_matches_oracle as compaction

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 3, 4, 5, 127, 128, 129])
@pytest.mark.parametrize("wide", [False, True])
def test_rollbacks_match_oracle(B, wide):
    m = umim()
    r = np.random.default_rng(B)
    lens = r.integers(16, 90, size=B)
    n_spans = np.where(r.random(B) < 0.6, r.integers(1, 5, size=B), 0)
    lens[0], n_spans[0] = (4100, 40) if wide else (60, 5)   # a 257-page table: the plan in a kernel of its own
    c = W.decode_case(400 + B, lens=lens, n_q_heads=2, n_kv_heads=1, head_dim=64, n_spans=list(n_spans), kmin=2, kmax=4,
                      spare_pages=2)
    g = case_to_dev(c, dev())
    status = m.new_status(dev())
    freed = m.umim_kv_rollback(g["pool"], g["bt"], g["lens"], g["offs"], g["st"], g["ln"], g["sk"], g["sv"],
                               dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    compare_rollback(g["pool"], g["bt"], g["lens"], freed, oracle_rollback(c))


@pytest.mark.parametrize("B", [127, 128, 129])
def test_compactions_match_oracle(B):
    compaction(B, B, 21, 512, 0.5)
