"""The rollback's plan and map at the edges of their blocks of spans and pages (1024 threads of up to 8 spans, 16 pages
and 256 keys per CTA), bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import case_to_dev, compare_rollback, dev, oracle_rollback, umim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lens,n_spans,kmin,kmax", [
    ([4096, 40], [255, 1], 2, 4), ([4096, 4096], [256, 257], 1, 4),
    ([2600], [1023], 1, 3), ([4200], [1025], 2, 4),                  # one and two spans a thread
    ([17000], [8192], 1, 2), ([17000], [8193], 1, 2),                # one and two passes
    ([3000], [1], 2900, 2900),                                       # a span over many pages
    ([257, 0, 256, 255], [1, 0, 1, 1], 1, 1),
    ([4096, 100], [4096, 100], 1, 1), ([4090, 1024, 1025], [1300, 7, 300], 2, 4),   # plan and map in one kernel: 256 pages
    ([4097, 64], [1300, 20], 2, 4),                                                  # and in two: 257
])
def test_span_counts_match_oracle(lens, n_spans, kmin, kmax):
    m = umim()
    c = W.decode_case(900 + sum(n_spans), lens=lens, n_q_heads=2, n_kv_heads=1, head_dim=64, n_spans=n_spans,
                      kmin=kmin, kmax=kmax, spare_pages=2)
    g = case_to_dev(c, dev())
    status = m.new_status(dev())
    freed = m.umim_kv_rollback(g["pool"], g["bt"], g["lens"], g["offs"], g["st"], g["ln"], g["sk"], g["sv"],
                               dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    compare_rollback(g["pool"], g["bt"], g["lens"], freed, oracle_rollback(c))


def test_more_spans_than_entries_are_refused():
    """More spans than a 256-page table has entries: invalid, nothing written."""
    m = umim()
    c = W.decode_case(77, lens=[4096], n_q_heads=2, n_kv_heads=1, head_dim=64, n_spans=[0])
    g = case_to_dev(c, dev())
    S = 5000
    i32 = lambda x: torch.as_tensor(x, dtype=torch.int32, device=dev())
    sur = torch.zeros((S, 1, 1, 64), dtype=torch.bfloat16, device=dev())
    status, before, table = m.new_status(dev()), g["pool"].clone(), g["bt"].clone()
    m.umim_kv_rollback(g["pool"], g["bt"], g["lens"], i32([0, S]), i32(np.arange(S) % 4096), i32(np.ones(S)), sur, sur,
                       dev_status=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 1
    assert torch.equal(g["pool"], before) and torch.equal(g["bt"], table) and int(g["lens"][0]) == 4096
