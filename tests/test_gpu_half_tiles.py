"""Many-row projections whose last round of CTA pairs hands out single weight tiles (256 x 128) beside or instead of pairs
of them: the same bits as whole items, and refreshes through every epilogue against the oracle."""
import dataclasses

import numpy as np
import pytest

import synth
from gpu_common import engine, requires_gpu
from test_gpu_gemm import _case
from test_gpu_many_rows import HD64, HD128, test_refresh_of_many_rows as check_refresh

PAIRS = 74      # CTA pairs of the GPU: one round


@requires_gpu
@pytest.mark.parametrize("pairs_of_tiles", [1, PAIRS // 2, PAIRS + 1, PAIRS + PAIRS // 2])
def test_single_tiles_give_the_bits_of_whole_items(pairs_of_tiles):
    """A weight's first rows give the same product whether its launch is one round of single tiles, whole items only, or a
    round of whole items and one of single tiles."""
    E = engine()
    M, N, K, whole = 200, 256 * (PAIRS + PAIRS // 2), 200, 256 * PAIRS      # 74 items: whole ones only
    xb, wb = _case(M, N, K, seed=11)
    x, w = E.bits_to_device(xb, "cuda"), E.bits_to_device(wb, "cuda")
    ref = E.debug_gemm(x, w[:whole], 1)
    n = 256 * pairs_of_tiles
    out = E.debug_gemm(x, w[:n], 1)
    m = min(n, whole)
    assert bool((out[:, :m] == ref[:, :m]).all())
    xf, wf = synth.bf16_bits_to_f32(xb).astype(np.float64), synth.bf16_bits_to_f32(wb[:n]).astype(np.float64)
    # fp32 accumulation of exact bf16 products, as in the other tests of this kernel
    assert np.abs(out.cpu().numpy() - xf @ wf.T).max() <= 2e-6 * (np.abs(xf) @ np.abs(wf).T).max()


@requires_gpu
@pytest.mark.parametrize("shape,P,L", [
    (dataclasses.replace(HD128, d_ffn=128 * (PAIRS + 5)), 100, 60),                 # gate/up: 79 items, the last five halved
    (dataclasses.replace(HD64, d_ffn=128 * (PAIRS + 22) - 48), 90, 150),            # 96 items; the last tile's features end early
    # QKV with RoPE: 84 items in seven row tiles, either head dim.  One layer: the helper's share of equal bf16 values of K and V
    # holds behind one layer of this width, not behind two (a difference of 1e-3 in a layer's output flips half of the roundings)
    (dataclasses.replace(HD64, n_layers=1, n_heads=16, d_model=1024), 1500, 100),
    (dataclasses.replace(HD128, n_layers=1, n_heads=8, d_model=1024), 1450, 110),
])
def test_refresh_through_single_tiles(shape, P, L):
    check_refresh(shape, P, L)
