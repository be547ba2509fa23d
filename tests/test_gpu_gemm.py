"""The tcgen05 weight-streaming GEMM against the oracle's matmul, through the C ABI."""
import numpy as np
import pytest
import torch

import synth
from gpu_common import engine, requires_gpu


def _case(M, N, K, seed):
    x = synth.normal_bf16(seed, 100, (M, K), 1.0)
    w = synth.normal_bf16(seed, 101, (N, K), 0.05)
    return x, w


@requires_gpu
@pytest.mark.parametrize("M,N,K,splits", [
    (32, 768, 256, 1),        # tiny-model QKV
    (32, 768, 256, 2),
    (16, 256, 688, 1),        # K tail: 688 = 10 * 64 + 48
    (16, 256, 688, 3),
    (64, 1376, 256, 0),       # N tail: 1376 = 10 * 128 + 96; 64-row tile
    (100, 2048, 256, 0),      # ragged rows inside a 128-row tile
    (128, 512, 1024, 4),
    (300, 640, 512, 0),       # many rows, odd number of weight tiles (5): single-CTA tiles of 128 rows, last ragged
    (300, 768, 512, 0),       # many rows, even number of weight tiles: CTA pairs, two 256-row tiles, second ragged
    (700, 1024, 688, 2),      # CTA pairs with a K split and a K tail; three row tiles, last ragged (188 rows)
    (129, 256, 64, 1),        # CTA pair, one k-block, one row in the second CTA's half
    (2305, 4060, 320, 1),     # 160 tiles for 74 CTA pairs: the third tile of a pair reuses the first accumulator; the second
                              # group has two row tiles, the last one a single row; the last weight tile 92 columns
    (2305, 4060, 320, 2),     # the same with a K split of unequal halves: 320 tiles of three and two k-blocks
    (1, 128, 64, 1),          # smallest
    (48, 2048, 2048, 0),
])
def test_gemm_matches_oracle(M, N, K, splits):
    E = engine()
    xb, wb = _case(M, N, K, seed=M + N + K)
    x = E.bits_to_device(xb, "cuda")
    w = E.bits_to_device(wb, "cuda")
    out = E.debug_gemm(x, w, splits).cpu().numpy().astype(np.float64)
    xf = synth.bf16_bits_to_f32(xb).astype(np.float64)
    wf = synth.bf16_bits_to_f32(wb).astype(np.float64)
    ref = xf @ wf.T
    scale = (np.abs(xf) @ np.abs(wf).T).max()
    err = np.abs(out - ref).max()
    assert err <= 2e-6 * scale, (err, scale)          # fp32 accumulation of exact bf16 products
    out2 = E.debug_gemm(x, w, splits).cpu().numpy().astype(np.float64)
    assert np.array_equal(out, out2)                   # fixed-order split reduction: bitwise repeatable


@requires_gpu
@pytest.mark.parametrize("M,N,K,splits,shift", [
    (129, 255, 64, 1, 0),       # two weight tiles, the last column of a 16-byte piece missing
    (300, 642, 512, 0, 0),      # rows start on 8-byte boundaries; the last piece holds two columns
    (257, 1021, 320, 2, 0),     # odd rows, a K split, one row in the second row tile
    (300, 768, 512, 2, 4),      # whole pieces, the partial sums' base 4 bytes off a 16-byte boundary
])
def test_many_rows_of_any_length_and_base(M, N, K, splits, shift):
    """CTA pairs store 16 bytes at a time where every row starts on such a boundary, single values elsewhere: nothing
    between, in front of or behind the rows is written."""
    import ctypes as C
    from paper_2511_21759_b200 import binding as B
    E = engine()
    xb, wb = _case(M, N, K, seed=M + N + K)
    x, w = E.bits_to_device(xb, "cuda"), E.pack_weight(E.bits_to_device(wb, "cuda"))
    room = max(splits, 16) * M * N * 4 + 1024
    scratch = torch.full((room + 512,), 0xA5, dtype=torch.uint8, device="cuda")
    out = torch.empty(M, N, dtype=torch.float32, device="cuda")
    at = 256 + shift
    B.check(B.lib().odb_debug_gemm(x.data_ptr(), w.data_ptr(), out.data_ptr(), scratch.data_ptr() + at, room, M, N, K,
                                   splits, C.c_void_p(torch.cuda.current_stream().cuda_stream)), "odb_debug_gemm")
    xf = synth.bf16_bits_to_f32(xb).astype(np.float64)
    wf = synth.bf16_bits_to_f32(wb).astype(np.float64)
    err = np.abs(out.cpu().numpy() - xf @ wf.T).max()
    assert err <= 2e-6 * (np.abs(xf) @ np.abs(wf).T).max()      # fp32 accumulation, as above
    if splits:
        raw = scratch.cpu().numpy()
        end = at + splits * M * N * 4
        status = at + (splits * M * N * 4 + 255) // 256 * 256   # the status word lies behind the partial sums
        assert (raw[:at] == 0xA5).all() and (raw[end:status] == 0xA5).all() and (raw[status + 4:] == 0xA5).all()


@requires_gpu
def test_gemm_garbage_rows_do_not_leak():
    """Rows of x beyond M are never read into the result: a 32-row tile fed 5 rows."""
    E = engine()
    xb, wb = _case(32, 256, 256, seed=9)
    big = E.bits_to_device(xb, "cuda")
    big[5:] = float("nan")
    w = E.bits_to_device(wb, "cuda")
    out = E.debug_gemm(big[:5], w, 1).cpu().numpy()
    ref = synth.bf16_bits_to_f32(xb[:5]).astype(np.float64) @ synth.bf16_bits_to_f32(wb).astype(np.float64).T
    assert np.isfinite(out).all() and np.abs(out - ref).max() < 1e-3
