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
    # CTA pairs, few rows: as many splits as leave 8 k-blocks each, while they fit one wave of 74 pairs
    (160, 3072, 1024, 2), (160, 1024, 1024, 2), (160, 1024, 2816, 5), (350, 1024, 2816, 5),
    (160, 6144, 2048, 3),                  # 24 tiles: three splits are one wave, four (8 k-blocks) would be two
    (1250, 3072, 1024, 1), (1250, 1024, 1024, 1), (1250, 1024, 2816, 3),   # many rows: the partials cost more
    (768, 4096, 4096, 3), (768, 4096, 12288, 3), (768, 12288, 4096, 1), (4096, 4096, 4096, 1),   # the 8B shape
    (300, 640, 1024, 2), (700, 1920, 2048, 3),   # odd numbers of weight tiles: single CTAs, 8 k-blocks per split
    (129, 256, 64, 1),                     # a single k-block
])
def test_k_splits_of_many_rows(M, N, K, splits):
    assert _rule("_ZN3odb16gemm_pick_splitsEiii", *[ctypes.c_int] * 3)(M, N, K) == splits


def test_k_splits_are_never_empty():
    pick = _rule("_ZN3odb16gemm_pick_splitsEiii", *[ctypes.c_int] * 3)
    for M in (1, 32, 128, 129, 256, 300, 768, 1118, 4096):
        for N in (64, 128, 255, 640, 1024, 3072, 12288):
            for nkb in list(range(1, 40)) + [64, 86, 192]:
                s = pick(M, N, 64 * nkb)
                assert 1 <= s <= max(1, nkb // 4) and -(-nkb // s) * (s - 1) < nkb, (M, N, nkb, s)
