"""The kernels that merge partial results - key splits of the attention, vocabulary tiles of the LM head - where their last
block or their last round of loads is not whole."""
import dataclasses

import pytest

from gpu_common import requires_gpu
from test_gpu_many_rows import HD64, HD128, test_refresh_of_many_rows as check_refresh


@requires_gpu
@pytest.mark.parametrize("shape,P,L", [
    (dataclasses.replace(HD64, n_heads=1, d_model=64), 1, 20),     # 21 (row, head) pairs: the third block of eight ends early
    (dataclasses.replace(HD128, n_heads=1, d_model=128), 3, 18),   # 21 pairs in blocks of four
    (dataclasses.replace(HD64, vocab=128 * 8 + 1), 5, 60),         # nine vocabulary tiles, one id in the last
    (dataclasses.replace(HD64, vocab=128 * 1025 + 3), 2, 33),      # two rounds of loads, the second with two tiles
])
def test_merges_at_their_edges(shape, P, L):
    v = shape.vocab
    check_refresh(dataclasses.replace(shape, mask_id=v - 1, eos_id=v - 2), P, L)


@requires_gpu
@pytest.mark.parametrize("rows,ffn", [(129, 13056), (200, 28672)])   # a down projection of 204 and 448 k-blocks: sixteen splits
def test_refresh_with_a_long_down_projection(rows, ffn):
    check_refresh(dataclasses.replace(HD64, n_layers=1, n_heads=16, d_model=1024, d_ffn=ffn), rows - 60, 60)
