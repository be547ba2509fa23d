"""The tensor-core attention where the order of sums is free (models without LM head) and launches have enough work items for it:
refreshes with head dim 64 around the edges of the 128-row items and 64-key tiles, steps of several copies with and without key
splits, in both row layouts, and batched steps of one copy."""
import dataclasses
import math

import numpy as np
import pytest
import torch

import synth
from gpu_common import bf16_bits_to_f64, engine, requires_gpu
from test_gpu_many_rows import HD64, HD128

HEADS = 32
SHAPE = dataclasses.replace(HD64, n_layers=1, n_heads=HEADS, d_model=64 * HEADS, d_ffn=256)


def rows(sess, name, hd=64):
    return torch.from_numpy(bf16_bits_to_f64(sess.debug_read(name))).view(-1, HEADS, hd)


def check(o, q, keys, vals, visible=None):
    s = torch.einsum("qhd,hkd->hqk", q, keys) / math.sqrt(q.shape[-1])
    if visible is not None:
        s = s.masked_fill(~visible[None], -math.inf)
    want = torch.einsum("hqk,hkd->qhd", torch.softmax(s, -1), vals).numpy()
    # the output is rounded to bf16 (half of the last of seven fraction bits: 2^-8 of the value at worst); fp32 scores and
    # sums, P as two bf16 terms: 2^-16 of the row's size
    rms = np.sqrt((want ** 2).mean(-1, keepdims=True))
    assert (np.abs(o.numpy() - want) <= 2.0 ** -8 * 1.01 * np.abs(want) + 2.0 ** -13 * rms).all()


@requires_gpu
@pytest.mark.parametrize("lens", [
    [(257, 64)],                          # three items (96 with 32 heads): the last has 65 rows; six key tiles, the last of one key
    [(320, 64)],                          # whole items and whole tiles
    [(100, 28), (1, 64), (70, 100)],      # one whole item, one of 65 rows, one and 42 rows
    [(1000, 70), (30, 33)],               # seventeen key tiles and one
])
def test_refresh(lens):
    E = engine()
    gm = E.Model.from_synth(SHAPE, seed=5, max_batch=len(lens), max_seq=max(p + n for p, n in lens), max_block=16, max_copies=1, with_lm_head=False)
    sess = E.Session(gm, poison=True)
    for i, (p, n) in enumerate(lens):
        sess.set_sequence(i, synth.sequence(5, i, p, n, SHAPE), p)
    sess.refresh_prefill(E.DecodeParams(block_len=16), 0)
    q, k, v, o = (rows(sess, x) for x in "qkvo")
    assert sess.status() == 0
    r0 = 0
    for p, n in lens:
        r = slice(r0, r0 + p + n)
        check(o[r], q[r], k[r].transpose(0, 1), v[r].transpose(0, 1))
        r0 += p + n
    assert r0 == len(o)
    sess.close(); gm.close()


@requires_gpu
@pytest.mark.parametrize("copies,decoded,block,batch,hd", [
    (4, 0, 32, 1, 64),       # one item per head: three cached key splits and the fresh one, two copies to a tile of fresh keys
    (4, 5, 24, 2, 64),       # 96 rows an item, copies across the tiles' edges
    (4, 0, 21, 1, 128),
    (8, 16, 24, 2, 128),     # the decoded-share layout in two items a sequence: the second sees copy 0's decoded rows in a tile of their own
    (8, 22, 32, 3, 64),      # in one
    (4, 0, 64, 5, 64),       # ten items per head: no key splits, the outputs are final
    (8, 44, 64, 5, 64),
    (1, 3, 37, 4, 128),      # one copy
    (1, 5, 17, 10, 64),
    (1, 60, 64, 8, 64),
])
def test_step_with_copies(copies, decoded, block, batch, hd):
    E = engine()
    lens = [(101 + 29 * (i % 4), max(block, 220 - 12 * i)) for i in range(batch)]
    shape = SHAPE if hd == 64 else dataclasses.replace(HD128, n_layers=1, n_heads=HEADS, d_model=128 * HEADS, d_ffn=256)
    gm = E.Model.from_synth(shape, seed=5, max_batch=batch, max_seq=max(p + n for p, n in lens), max_block=block, max_copies=8, with_lm_head=False)
    sess = E.Session(gm, poison=True)
    for i, (p, n) in enumerate(lens):
        x = synth.sequence(5, i, p, n, shape)
        at = np.random.default_rng(i).permutation(block)[:decoded]
        x[p + at] = 7 + at                                             # ids other than [MASK] and [EOS]
        sess.set_sequence(i, x, p)
    par = E.DecodeParams(block_len=block, n_copies=copies, alp=False)
    sess.refresh_prefill(par, 0)
    sess.unmask_accept(par, True)
    sess.block_decode_step(par)
    copy, pos = sess.debug_read("row_copy"), sess.debug_read("row_pos")
    # the rows are in sequence order, copy 0 first; consecutive blocks do not follow one another
    seq = np.cumsum(np.r_[1, (copy[1:] == 0) & ((copy[:-1] != 0) | (pos[1:] != pos[:-1] + 1))]) - 1
    q, k, v, o = (rows(sess, x, hd) for x in "qkvo")
    assert sess.status() == 0
    kv = sess.kv.view(torch.bfloat16).view(batch, 2, HEADS, -1, hd).double().cpu()
    for i, (p, n) in enumerate(lens):
        r = np.flatnonzero(seq == i)
        x = sess.get_tokens(i)
        sees = copy[r][:, None] == copy[r][None, :]
        if len(r) < copies * block:
            sees |= ((copy[r] == 0) & (x[pos[r]] != shape.mask_id))[None, :]
        out = [j for j in range(p + n) if not p <= j < p + block]
        keys, vals = (torch.cat([kv[i, j][:, out], f[r].transpose(0, 1)], 1) for j, f in ((0, k), (1, v)))
        check(o[r], q[r], keys, vals, torch.cat([torch.ones(len(r), len(out), dtype=torch.bool), torch.from_numpy(sees)], 1))
    sess.close(); gm.close()


@requires_gpu
@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("log2_gain", [11, 17, 40])     # scores of about 2^22, 2^34 and 2^80 in the log2 domain
def test_refresh_with_scores_far_beyond_the_range_of_their_differences(hd, log2_gain):
    """Every row sees one key alone: its output is that key's v."""
    E = engine()
    shape = SHAPE if hd == 64 else dataclasses.replace(HD128, n_layers=1, n_heads=HEADS, d_model=128 * HEADS, d_ffn=256)
    p, n = 257, 64
    kw = dict(max_batch=1, max_seq=p + n, max_block=16, max_copies=1, with_lm_head=False)
    gm = E.Model.from_synth(shape, seed=5, **kw)
    t = dict(gm.t)
    gm.close()
    t["norm1"] = [t["norm1"][0] * 2.0 ** log2_gain]
    gm = E.Model(shape, t, **kw)
    sess = E.Session(gm, poison=True)
    sess.set_sequence(0, synth.sequence(5, 0, p, n, shape), p)
    sess.refresh_prefill(E.DecodeParams(block_len=16), 0)
    q, k, v, o = (rows(sess, x, hd) for x in "qkvo")
    assert sess.status() == 0
    s = torch.einsum("qhd,khd->hqk", q, k)
    # fp32 sums of hd products: 2^-24 of the sum of their sizes for each addition
    off = hd * 2.0 ** -23 * torch.einsum("qhd,khd->hqk", q.abs(), k.abs()).amax(-1)
    best = s.topk(2, -1)
    # the runner-up's weight vanishes where even the computed scores lie 2^5 apart in the log2 domain
    alone = best.values[..., 0] - best.values[..., 1] > 2 * off + 2.0 ** 5 * math.sqrt(hd) / math.log2(math.e)
    assert alone.double().mean() > 0.9
    want = torch.gather(v.transpose(0, 1), 1, best.indices[..., :1].expand(-1, -1, hd)).transpose(0, 1)
    seen = alone.T[..., None].expand_as(o)
    # one P alone, in two bf16 terms: 2^-16, then the rounding to bf16; the others' P below 2^-32 together with 320 of them
    assert ((o - want).abs() <= 2.0 ** -8 * want.abs() + 2.0 ** -20 * want.abs().amax())[seen].all()
    sess.close(); gm.close()
