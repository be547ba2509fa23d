"""The host-side rules that choose how a launch is divided, on a machine without a GPU: the library's own C++ functions,
called through their exported names."""
import ctypes

import pytest


def _rule(name, *argtypes):
    from paper_2511_21759_b200 import binding as B
    f = getattr(B.lib(), name)
    f.argtypes, f.restype = argtypes, ctypes.c_int
    return f


@pytest.mark.parametrize("items,hd,refresh,splits", [
    (4, 64, False, 8), (37, 64, False, 8),                          # never more than eight
    (80, 64, False, 4), (128, 64, False, 3), (192, 64, False, 2), (256, 64, False, 2),   # rounded up: three CTAs fit an SM
    (296, 64, False, 1), (297, 64, False, 1), (5000, 64, False, 1),
    (96, 128, False, 3), (128, 128, False, 2), (192, 128, False, 1), (1024, 128, False, 1),   # rounded down: two fit
    (128, 128, True, 3), (128, 64, True, 3), (300, 128, True, 1),   # a refresh rounds up with either
])
def test_key_splits_of_the_attention(items, hd, refresh, splits):
    assert _rule("_ZN3odb20attention_key_splitsEiib", ctypes.c_int, ctypes.c_int, ctypes.c_bool)(items, hd, refresh) == splits


@pytest.mark.parametrize("M,N,K,splits", [
    (200, 1024, 13056, 16), (200, 1024, 28672, 16), (129, 64, 1 << 17, 16),   # the consumers add up sixteen partials at most
    (256, 2304, 12480, 15), (256, 2304, 13056, 16), (768, 4096, 4096, 3),     # many rows: at least 12 k-blocks each
    (32, 4096, 12288, 9), (128, 1024, 28672, 16),                             # up to 128 rows: one wave
])
def test_k_splits_of_a_projection(M, N, K, splits):
    assert _rule("_ZN3odb16gemm_pick_splitsEiii", ctypes.c_int, ctypes.c_int, ctypes.c_int)(M, N, K) == splits


@pytest.mark.parametrize("M,N,K,splits", [
    (768, 4096, 4096, 3), (900, 4096, 4096, 1), (900, 4096, 12288, 1), (1200, 4096, 12288, 4),   # rounds of the pairs against sums
    (512, 2048, 5504, 4), (2000, 2048, 2048, 1), (25568, 4096, 12288, 1), (2600, 4096, 4096, 1), (2800, 2048, 5504, 1),
    (200, 1024, 1024, 2), (200, 1024, 960, 1), (200, 256, 688, 1),                               # at least eight k-blocks each
    (129, 256, 1 << 17, 16),                                                                     # sixteen partials at most
])
def test_k_splits_of_a_many_row_forward(M, N, K, splits):
    assert _rule("_ZN3odb16gemm_rows_splitsEiii", ctypes.c_int, ctypes.c_int, ctypes.c_int)(M, N, K) == splits
