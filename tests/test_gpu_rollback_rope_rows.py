"""Rotation of two rows at once (rotary dims up to 64, both head dims): pages whose moved entries begin and end at every
slot, so that rows are left over from the pairs, and rotary dims that leave lanes without a pair of elements; the
comparison of test_gpu_rollback_rope."""
import pytest

from test_gpu_rollback_rope import test_rope_rollback_matches_oracle as _matches_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed,lens,hkv,D,layers,rd,coverage", [
    (175, list(range(3, 90, 3)), 1, 64, 1, 64, 0.2), (176, list(range(5, 90, 4)), 2, 64, 2, 16, 0.5),
    (177, list(range(3, 90, 5)), 1, 128, 1, 64, 0.3), (178, [400, 77], 1, 128, 1, 32, 0.1),
    (179, [1200], 2, 64, 1, 48, 0.6), (180, [600, 41], 2, 128, 1, 80, 0.3),   # 80: one row at a time
])
def test_rows_of_a_pair(seed, lens, hkv, D, layers, rd, coverage):
    _matches_oracle(seed, lens, hkv, D, layers, rd, coverage)
