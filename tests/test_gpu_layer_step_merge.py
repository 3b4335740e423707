"""The per-layer step's merges of segments split over warps, at every number of pieces about the limit (25) from
which the warps of a CTA share a merge, and over hundreds of pieces, against the oracle (test_gpu_layer_step's
comparison): rows of G = 1, 5, 7 and 16 query heads leave remainders of the four rows taken together."""
import pytest

from test_gpu_layer_step import _run_steps

pytestmark = pytest.mark.gpu

# 16-entry pages, one to a warp while they are fewer than the GPU's warps: 22 to 28 pieces, and short ones
ABOUT = [340, 372, 386, 403, 419, 436, 60, 5]


@pytest.mark.parametrize("seed,lens,hq,hkv,d", [
    (71, ABOUT, 7, 1, 128), (72, ABOUT, 16, 1, 64), (73, ABOUT, 10, 2, 64), (74, ABOUT, 2, 2, 128),
    (75, [12000], 16, 1, 128), (76, [29000, 17], 28, 4, 64),
])
def test_split_segments_match_oracle(seed, lens, hq, hkv, d):
    _run_steps(seed, lens, hq, hkv, d, 2, 2, p_merge=1.0)
