"""The mma.sync attention where whole key tiles and tiles with a mask meet: refreshes with head dim 64 around multiples of 64
keys, and a batched step whose keys are not split, around a block that ends on and off a tile."""
import dataclasses
import math

import numpy as np
import pytest
import torch

import synth
from gpu_common import bf16_bits_to_f64, engine, requires_gpu
from test_gpu_many_rows import HD64, HD128, test_refresh_of_many_rows as check_refresh


@requires_gpu
@pytest.mark.parametrize("P,L", [(65, 64), (64, 65), (92, 100), (100, 93), (200, 120), (255, 257)])
def test_refresh_around_whole_tiles(P, L):
    check_refresh(dataclasses.replace(HD64, n_layers=1), P, L)


@requires_gpu
@pytest.mark.parametrize("shape,batch", [
    (dataclasses.replace(HD64, n_layers=1, n_heads=32, d_model=2048, d_ffn=256), 10),    # 320 items for 296 slots: no key splits
    (dataclasses.replace(HD128, n_layers=1, n_heads=32, d_model=4096, d_ffn=256), 5),    # 160: none with head dim 128
])
def test_step_without_key_splits(shape, batch):
    E = engine()
    lens = [(64 * (1 + i % 3) - (i % 4) * 5, 96 - 7 * i) for i in range(batch)]          # blocks start and end on and off tiles
    gm = E.Model.from_synth(shape, seed=5, max_batch=batch, max_seq=max(p + n for p, n in lens), max_block=16, max_copies=1)
    sess = E.Session(gm, poison=True)
    for i, (p, n) in enumerate(lens):
        sess.set_sequence(i, synth.sequence(5, i, p, n, shape), p)
    par = E.DecodeParams(block_len=16)
    sess.refresh_prefill(par, 0)
    sess.unmask_accept(par, True)
    sess.block_decode_step(par)
    q, k, v, o = (torch.from_numpy(bf16_bits_to_f64(sess.debug_read(x))).view(-1, shape.n_heads, shape.head_dim) for x in "qkvo")
    assert sess.status() == 0 and len(q) == 16 * batch
    kv = sess.kv.view(torch.bfloat16).view(batch, 2, shape.n_heads, -1, shape.head_dim).double().cpu()
    for i, (p, n) in enumerate(lens):
        r = slice(16 * i, 16 * i + 16)
        out = [j for j in range(p + n) if not p <= j < p + 16]
        keys, vals = (torch.cat([kv[i, j][:, out], x[r].transpose(0, 1)], 1) for j, x in ((0, k), (1, v)))
        s = torch.einsum("qhd,hkd->hqk", q[r], keys) / math.sqrt(shape.head_dim)
        want = torch.einsum("hqk,hkd->qhd", torch.softmax(s, -1), vals).numpy()
        got = o[r].numpy()
        # the output is rounded to bf16 (half of the last of seven fraction bits: 2^-8 of the value at worst); fp32 scores and
        # sums, P as two bf16 terms: 2^-16 of the row's size
        rms = np.sqrt((want ** 2).mean(-1, keepdims=True))
        assert (np.abs(got - want) <= 2.0 ** -8 * 1.01 * np.abs(want) + 2.0 ** -13 * rms).all(), i
    sess.close(); gm.close()
