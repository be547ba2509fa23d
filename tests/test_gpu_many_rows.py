"""The many-row projections (more than 128 rows) at the edges of their tiles, in the product mode (no logits): the
refresh's confidences, greedy tokens and K/V against the oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import synth
from oracle import odb_oracle as O
from oracle.inputs import model_from_synth
from gpu_common import engine, requires_gpu, bf16_bits_to_f64, logits_close

# d_ffn 736: 12 gate/up tiles, the last half empty; vocabulary 1980: 16 tiles, the last with 60 ids, [MASK] and [EOS] in it
HD128 = dataclasses.replace(synth.TINY_HD128, d_ffn=736, vocab=1980, mask_id=1979, eos_id=1978)
HD64 = dataclasses.replace(synth.TINY, d_ffn=736, vocab=1980, mask_id=1700, eos_id=1978)


@requires_gpu
@pytest.mark.parametrize("shape,P,L", [
    (HD128, 1, 128),      # one row beyond the first CTA's 128
    (HD128, 100, 156),    # one whole 256-row tile
    (HD64, 60, 197),      # one row in the second tile
    (HD128, 37, 348),     # second tile: one row in the second CTA's half
    (HD64, 301, 230),     # three tiles, the last ragged; 230 response rows through the LM head
    (dataclasses.replace(HD64, n_heads=3, d_model=192), 150, 90),   # an odd number of heads
])
def test_refresh_of_many_rows(shape, P, L):
    E = engine()
    om = model_from_synth(shape, seed=5)
    gm = E.Model.from_synth(shape, seed=5, max_batch=1, max_seq=P + L, max_block=16, max_copies=1)
    sess = E.Session(gm, poison=True)
    x0 = synth.sequence(5, 0, P, L, shape)
    sess.set_sequence(0, x0, P)
    sess.refresh_prefill(E.DecodeParams(block_len=16), 0)
    conf, tok = sess.debug_read("conf"), sess.debug_read("tok")
    k, v = (bf16_bits_to_f64(sess.debug_read(n)) for n in "kv")
    assert sess.status() == 0
    cache, oconf, otok, ologits = O.refresh_prefill(om, x0, P + L, P, return_logits=True)
    # confidences of the N(0, 0.02) models move like their logits: the 2e-2 of the other refresh tests
    assert conf.shape == (L,) and np.allclose(conf, oconf, rtol=2e-2)
    ologits[:, shape.mask_id] = -np.inf
    chosen = np.take_along_axis(ologits, tok[:, None].astype(np.int64), 1)[:, 0]
    rms = np.sqrt((np.delete(ologits, shape.mask_id, 1) ** 2).mean(1))
    assert (ologits.max(1) - chosen <= 2 * 2e-2 * rms).all()      # a token other than the oracle's only where the two tie
    for got, want in ((k, cache.k[-1]), (v, cache.v[-1])):
        ok, worst = logits_close(got, want.reshape(P + L, -1), 4e-2)
        assert ok, worst
        assert (got == want.reshape(P + L, -1)).mean() > 0.7
    kv = sess.kv.view(torch.bfloat16).view(1, shape.n_layers, 2, shape.n_heads, P + L, shape.head_dim).float().cpu().numpy()
    for j, got in ((0, k), (1, v)):                               # the cache holds what the fresh rows hold
        assert np.array_equal(kv[0, -1, j].transpose(1, 0, 2).reshape(P + L, -1), got)
    sess.close(); gm.close()


@requires_gpu
def test_refresh_of_two_sequences_beyond_one_tile_per_pair():
    """3120 rows of two sequences, 13 row tiles: the QKV projection hands out 156 tiles (head dim 64, more than two per
    CTA pair), gate/up 78, and the second sequence's rows go to its own part of the cache, in every layer."""
    E = engine()
    shape = dataclasses.replace(HD64, n_heads=16, d_model=1024)
    lens = [(1500, 220), (1161, 239)]
    longest = max(p + n for p, n in lens)
    om = model_from_synth(shape, seed=5)
    gm = E.Model.from_synth(shape, seed=5, max_batch=2, max_seq=longest, max_block=16, max_copies=1)
    sess = E.Session(gm, poison=True)
    for i, (p, n) in enumerate(lens):
        sess.set_sequence(i, synth.sequence(5, i, p, n, shape), p)
    sess.refresh_prefill(E.DecodeParams(block_len=16), 0)
    conf = sess.debug_read("conf")
    kv = sess.kv.view(torch.bfloat16).view(2, shape.n_layers, 2, shape.n_heads, longest, shape.head_dim).float().cpu().numpy()
    assert sess.status() == 0
    at = 0
    for i, (p, n) in enumerate(lens):
        cache, oconf, _ = O.refresh_prefill(om, synth.sequence(5, i, p, n, shape), p + n, p)
        assert np.allclose(conf[at:at + n], oconf, rtol=2e-2)
        at += n
        for l in range(shape.n_layers):
            for j, want in ((0, cache.k[l]), (1, cache.v[l])):
                got = kv[i, l, j, :, : p + n].transpose(1, 0, 2).reshape(p + n, -1)
                ok, worst = logits_close(got, want.reshape(p + n, -1), 4e-2)
                assert ok, (i, l, j, worst)
    assert at == len(conf)
    sess.close(); gm.close()


@requires_gpu
@pytest.mark.parametrize("L", [60, 230])      # 97 rows: one row per block of the first norm; 267: four
def test_an_embedding_table_on_any_4_byte_boundary(L):
    """A table that starts 4 bytes behind an 8-byte boundary is read in halves: the same bits."""
    E = engine()
    P, x0 = 37, synth.sequence(5, 0, 37, L, HD64)
    par = E.DecodeParams(block_len=16)
    got = []
    for shift in (0, 2):
        gm = E.Model.from_synth(HD64, seed=5, max_batch=1, max_seq=P + L, max_block=16, max_copies=1)
        if shift:
            t = dict(gm.t)
            table = torch.empty(t["embed"].numel() + shift, dtype=torch.bfloat16, device="cuda")[shift:].view_as(t["embed"])
            table.copy_(t["embed"])
            t["embed"] = table
            assert table.data_ptr() % 8 == 4
            gm.close()
            gm = E.Model(HD64, t, max_batch=1, max_seq=P + L, max_block=16, max_copies=1)
        sess = E.Session(gm, poison=True)
        sess.set_sequence(0, x0, P)
        sess.refresh_prefill(par, 0)
        refreshed = sess.debug_read("hidden")
        sess.unmask_accept(par, True)
        sess.block_decode_step(par)
        got.append((refreshed, sess.debug_read("hidden"), sess.debug_read("conf"), sess.debug_read("tok")))
        assert sess.status() == 0
        sess.close(); gm.close()
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.array_equal(a, b)
