"""SwiGLU in the gate/up projections' epilogues over the whole range of gates: where e^-gate overflows, where the quotient is too small
for a normal number, and large positive ones.  Every row is the same known vector, every gate a chosen value."""
import ctypes
import dataclasses

import numpy as np
import pytest
import torch

import synth
from gpu_common import engine, requires_gpu

D, F = 256, 128
GATES = [-3e38, -1e30, -300, -104, -89, -88.5, -88, -87.5, -87, -60, -20, -3.25, -1, -2.0 ** -20, -1e-30, 0, 1e-30, 2.0 ** -12, 0.5, 1.75, 20, 87, 89, 300, 1e5, 1e30]


@requires_gpu
@pytest.mark.parametrize("rows", [5, 40, 100, 300])           # the three row tiles of few rows, the kernel of many
def test_swiglu_over_all_gates(rows):
    E = engine()
    shape = dataclasses.replace(synth.TINY, n_layers=1, d_model=D, n_heads=4, d_ffn=F, vocab=32, mask_id=31, eos_id=30, rms_eps=0.0)

    def dev(x):
        return torch.tensor(x, device="cuda", dtype=torch.bfloat16)

    gate = torch.tensor([GATES[i % len(GATES)] for i in range(F)]).to(torch.bfloat16)      # exact in bf16 from here on
    wgu = torch.zeros(2 * F, D, dtype=torch.bfloat16)
    wgu[:F, 0], wgu[F:, 1] = gate, 1.5                          # the normalised row is all ones: gate i, up 1.5
    wd = torch.zeros(D, F, dtype=torch.bfloat16)
    wd[torch.arange(F), torch.arange(F)] = 1
    ones = torch.ones(D, device="cuda")
    zeros = torch.zeros(4 * D, D, device="cuda", dtype=torch.bfloat16)
    gm = E.Model(shape, {"embed": dev(np.ones((32, D))), "final_norm": ones, "norm1": [ones], "norm2": [ones], "lm_head": None,
                         "wqkv": [E.pack_weight(zeros[: 3 * D].contiguous())], "wo": [E.pack_weight(zeros[:D].contiguous())],
                         "wgu": [E.pack_gate_up(wgu.cuda())], "wd": [E.pack_weight(wd.cuda())]},
                 max_batch=1, max_seq=rows, max_block=4, max_copies=1, with_lm_head=False)
    sess = E.Session(gm, poison=True)
    sess.set_sequence(0, synth.sequence(1, 0, rows - 4, 4, shape), rows - 4)
    sess.refresh_prefill(E.DecodeParams(block_len=4), 0)
    got = sess.debug_read("hidden").astype(np.float64) - 1.0    # the embedding is all ones
    assert sess.status() == 0 and got.shape == (rows, D)
    c = gate.double().numpy()
    with np.errstate(over="ignore"):
        want = c / (1.0 + np.exp(-c)) * 1.5
    # bf16 of the product, and the rounding of 1 + it in fp32
    assert (np.abs(got[:, :F] - want) <= 2.0 ** -8 * np.abs(want) + 2.0 ** -23 * (1 + np.abs(want))).all()
    assert (got[:, F:] == 0).all()
    sess.close(); gm.close()


@requires_gpu
def test_the_corrected_quotient_is_the_division_bit_for_bit():
    """All 2^32 gates, NaN and infinities among them: -0 alone, whose quotient loses its sign, differs."""
    engine()
    from paper_2511_21759_b200 import binding as B
    f = B.lib()._ZN3odb16launch_silu_bitsEPyP11CUstream_st
    f.argtypes, f.restype = (ctypes.c_void_p, ctypes.c_void_p), ctypes.c_int
    out = torch.tensor([0, (1 << 63) - 1], dtype=torch.int64, device="cuda")
    assert f(out.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    assert out.tolist() == [1, 1 << 31]
