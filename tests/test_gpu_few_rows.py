"""The projections of up to 128 rows at the edges of their tiles and stage rings: plain products against the oracle's
matmul, and refreshes whose gate/up and LM-head epilogues run in groups of warps, in the product mode, against the oracle."""
import dataclasses

import numpy as np
import pytest

import synth
from gpu_common import engine, requires_gpu
from test_gpu_gemm import _case
from test_gpu_many_rows import HD64, HD128, test_refresh_of_many_rows as check_refresh


@requires_gpu
@pytest.mark.parametrize("M", [32, 33, 65])                        # 32-, 64- and 128-row tiles
@pytest.mark.parametrize("kb", [1, 2, 3, 4, 5, 6, 7, 9, 16])       # k-blocks against rings of 3 to 5 stages
def test_product_over_the_stage_rings(M, kb):
    E = engine()
    N, K = 256, 64 * kb - 8                                        # the last k-block is not whole
    xb, wb = _case(M, N, K, seed=M + K)
    out = E.debug_gemm(E.bits_to_device(xb, "cuda"), E.bits_to_device(wb, "cuda"), 1).cpu().numpy().astype(np.float64)
    xf, wf = synth.bf16_bits_to_f32(xb).astype(np.float64), synth.bf16_bits_to_f32(wb).astype(np.float64)
    # fp32 accumulation of exact bf16 products, as in the other tests of this kernel
    assert np.abs(out - xf @ wf.T).max() <= 2e-6 * (np.abs(xf) @ np.abs(wf).T).max()


@requires_gpu
@pytest.mark.parametrize("shape,P,L", [
    (HD64, 1, 32),                                                 # 33 rows: 64-row tiles, 32 rows through the LM head
    (HD64, 7, 57),                                                 # 64 rows; 57 in the LM head: the second group's last rows are missing
    (HD128, 0, 65),                                                # 128-row tiles with one row behind the first half
    (HD64, 28, 97),                                                # one row for the last of the LM head's four groups
    (HD128, 0, 128),                                               # whole tiles
    (dataclasses.replace(HD64, n_heads=1, d_model=64), 3, 120),    # one k-block
    (dataclasses.replace(HD64, n_heads=7, d_model=448), 3, 70),    # seven
])
def test_refresh_of_few_rows(shape, P, L):
    check_refresh(shape, P, L)


@requires_gpu
@pytest.mark.parametrize("M", [1, 16, 17, 48, 49, 80, 81, 96, 97, 112, 113, 128])    # around the steps of sixteen rows that are loaded
@pytest.mark.parametrize("kb,splits", [(1, 1), (9, 1), (9, 2)])
def test_product_of_as_many_rows_as_there_are(M, kb, splits):
    E = engine()
    N, K = 384, 64 * kb
    xb, wb = _case(M, N, K, seed=M + K)
    out = E.debug_gemm(E.bits_to_device(xb, "cuda"), E.bits_to_device(wb, "cuda"), splits).cpu().numpy().astype(np.float64)
    xf, wf = synth.bf16_bits_to_f32(xb).astype(np.float64), synth.bf16_bits_to_f32(wb).astype(np.float64)
    # fp32 accumulation of exact bf16 products, as in the other tests of this kernel
    assert np.abs(out - xf @ wf.T).max() <= 2e-6 * (np.abs(xf) @ np.abs(wf).T).max()


@requires_gpu
@pytest.mark.parametrize("rows", [16, 17, 48, 80, 81, 96, 112, 113])
def test_refresh_of_as_many_rows_as_there_are(rows):
    check_refresh(HD64, rows - rows // 2, rows // 2)
