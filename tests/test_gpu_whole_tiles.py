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


@requires_gpu
@pytest.mark.parametrize("copies,decoded", [(4, 0), (8, 22)])          # 22 of 32 decoded: the decoded-share layout
@pytest.mark.parametrize("heads", [4, 32])                             # one cached tile per key split, and two
def test_step_with_copies_around_whole_tiles(heads, copies, decoded):
    """101 keys in front of the block and 232 behind it: a tile that holds keys of both sides is followed by whole ones that
    start off a multiple of 64, and the last ends early.  Every row sees its own copy's rows; in the decoded-share layout
    copy 0's decoded ones too."""
    E = engine()
    shape = dataclasses.replace(HD64, n_layers=1, n_heads=heads, d_model=64 * heads)
    P, L, block = 101, 264, 32
    gm = E.Model.from_synth(shape, seed=5, max_batch=1, max_seq=P + L, max_block=block, max_copies=8)
    sess = E.Session(gm, poison=True)
    x0 = synth.sequence(5, 0, P, L, shape)
    at = np.random.default_rng(1).permutation(block)[:decoded]
    x0[P + at] = 7 + at                                                # ids other than [MASK] and [EOS]
    sess.set_sequence(0, x0, P)
    par = E.DecodeParams(block_len=block, n_copies=copies, alp=False)
    sess.refresh_prefill(par, 0)
    sess.unmask_accept(par, True)
    sess.block_decode_step(par)
    x, copy, pos = sess.get_tokens(0), sess.debug_read("row_copy"), sess.debug_read("row_pos")
    q, k, v, o = (torch.from_numpy(bf16_bits_to_f64(sess.debug_read(n))).view(-1, heads, 64) for n in "qkvo")
    assert sess.status() == 0 and len(set(copy.tolist())) == copies
    share = len(copy) < copies * block
    assert share == (copies == 8)
    sees = copy[:, None] == copy[None, :]
    if share:
        sees |= ((copy == 0) & (x[pos] != shape.mask_id))[None, :]
    kv = sess.kv.view(torch.bfloat16).view(2, heads, -1, 64).double().cpu()
    out = [j for j in range(P + L) if not P <= j < P + block]
    keys, vals = (torch.cat([kv[j][:, out], r.transpose(0, 1)], 1) for j, r in ((0, k), (1, v)))
    s = torch.einsum("qhd,hkd->hqk", q, keys) / math.sqrt(64)
    s[:, :, len(out):].masked_fill_(~torch.from_numpy(sees)[None], -math.inf)
    want = torch.einsum("hqk,hkd->qhd", torch.softmax(s, -1), vals).numpy()
    # the bound of the test above
    rms = np.sqrt((want ** 2).mean(-1, keepdims=True))
    assert (np.abs(o.numpy() - want) <= 2.0 ** -8 * 1.01 * np.abs(want) + 2.0 ** -13 * rms).all()
    sess.close(); gm.close()
