"""A refresh with LM head runs the last layer's gate/up and down projections over the response rows only.  The same
token ids with no prompt make every row a response row, so that every projection runs over all of them: the
confidences and tokens of the rows both have are the same, and the keys and values too."""
import dataclasses

import numpy as np
import pytest
import torch

import synth
from gpu_common import engine, requires_gpu
from test_gpu_many_rows import HD64, HD128

ONE = dataclasses.replace(HD64, n_layers=1)


def _refresh(E, gm, seqs, prompts, block=0):
    sess = E.Session(gm, poison=True)
    for i, (x, p) in enumerate(zip(seqs, prompts)):
        sess.set_sequence(i, x, p)
    sess.refresh_prefill(E.DecodeParams(block_len=16), block)
    out = sess.debug_read("conf"), sess.debug_read("tok"), sess.debug_read("o"), sess.kv.clone()
    assert sess.status() == 0
    sess.close()
    return out


@requires_gpu
@pytest.mark.parametrize("shape,lens", [
    (HD128, [(500, 140)]),                    # three row tiles, then one
    (HD64, [(301, 270)]),                     # three tiles, then two with 270 rows
    (ONE, [(300, 40)]),                       # 40 rows in the kernel of 340
    (HD128, [(250, 7)]),                      # one row tile of seven rows
    (HD64, [(60, 31)]),                       # 128-row tiles, then 32-row ones
    (HD64, [(600, 16), (1, 150), (263, 40)]),                        # three sequences: their rows are gathered
    (dataclasses.replace(HD64, n_heads=3, d_model=192), [(200, 90), (150, 33)]),   # three weight tiles: single-CTA tiles of 128 rows
    (dataclasses.replace(HD128, n_heads=8, d_model=1024, n_layers=1), [(650, 130), (100, 200)]),   # O without K splits; 330 rows
])
def test_last_layer_over_the_response_rows(shape, lens):
    E = engine()
    gm = E.Model.from_synth(shape, seed=5, max_batch=len(lens), max_seq=max(p + n for p, n in lens), max_block=16, max_copies=1)
    seqs = [synth.sequence(5, i, p, n, shape) for i, (p, n) in enumerate(lens)]
    conf, tok, o, kv = _refresh(E, gm, seqs, [p for p, _ in lens])
    aconf, atok, ao, akv = _refresh(E, gm, seqs, [0] * len(lens))
    gm.close()
    at = np.cumsum([0] + [p + n for p, n in lens])
    rows = np.concatenate([np.arange(at[i] + p, at[i + 1]) for i, (p, _) in enumerate(lens)])
    assert np.array_equal(tok, atok[rows]) and np.array_equal(o, ao) and torch.equal(kv, akv)
    if len(rows) >= 256:                      # the final norm and the LM head run as the same kernels
        assert np.array_equal(conf, aconf[rows])
    else:
        # the final norm's sum of squares and the LM head's sum of exponentials in another order: a few 2^-24 of logits below 8 in
        # every term (1e-6), and at most 2^-24 for each of 1980 terms (1.2e-4)
        assert np.allclose(conf, aconf[rows], rtol=1.3e-4, atol=0)


@requires_gpu
@pytest.mark.parametrize("shape,lens", [
    (HD128, [(500, 140)]),                                           # O with K splits, one sequence
    (HD64, [(600, 16), (1, 150), (263, 40)]),                        # several
    (dataclasses.replace(HD64, n_heads=3, d_model=192), [(200, 90), (150, 33)]),
    (dataclasses.replace(HD128, n_heads=8, d_model=1024, n_layers=1), [(650, 130), (100, 200)]),   # O adds to the stream itself
    (HD64, [(60, 31)]),                                              # up to 128 rows
])
def test_residual_stream_of_the_prompt_rows_holds_the_last_attention_block(shape, lens):
    """The last layer's FFN reaches the rows with logits only, its attention block every row: with a last down projection of
    zeros, a refresh in which every row is a response row leaves that residual stream in all of them."""
    E = engine()
    gm = E.Model.from_synth(shape, seed=5, max_batch=len(lens), max_seq=max(p + n for p, n in lens), max_block=16, max_copies=1)
    sess = E.Session(gm, poison=True)

    def hidden(prompts):
        for i, ((p, n), at) in enumerate(zip(lens, prompts)):
            sess.set_sequence(i, synth.sequence(5, i, p, n, shape), at)
        sess.refresh_prefill(E.DecodeParams(block_len=16), 0)
        out = sess.debug_read("hidden")
        sess.unmask_accept(E.DecodeParams(block_len=16), True)
        return out

    got = hidden([p for p, _ in lens])
    gm.t["wd"][-1].zero_()
    want = hidden([0] * len(lens))
    assert sess.status() == 0
    at = np.cumsum([0] + [p + n for p, n in lens])
    rows = np.concatenate([np.arange(at[i], at[i] + p) for i, (p, _) in enumerate(lens)])
    assert len(rows) and np.isfinite(want).all() and np.array_equal(got[rows], want[rows])
    sess.close(); gm.close()


@requires_gpu
@pytest.mark.parametrize("lens,block", [
    ([(300, 2100)], 0),                       # 2100 rows through the LM head: a second chunk of 52
    ([(200, 1100), (150, 1000)], 0),          # gathered
    ([(500, 140)], 2),                        # the rows with logits start two blocks behind the prompt
    ([(263, 90), (1, 200)], 1),
])
def test_rows_with_logits_in_chunks_and_behind_later_blocks(lens, block):
    E = engine()
    shape = dataclasses.replace(HD64, n_layers=1)
    gm = E.Model.from_synth(shape, seed=5, max_batch=len(lens), max_seq=max(p + n for p, n in lens), max_block=16, max_copies=1)
    seqs = [synth.sequence(5, i, p, n, shape) for i, (p, n) in enumerate(lens)]
    conf, tok, o, kv = _refresh(E, gm, seqs, [p for p, _ in lens], block)
    aconf, atok, ao, akv = _refresh(E, gm, seqs, [0] * len(lens))
    gm.close()
    at = np.cumsum([0] + [p + n for p, n in lens])
    rows = np.concatenate([np.arange(at[i] + p + 16 * block, at[i + 1]) for i, (p, _) in enumerate(lens)])
    assert len(conf) == len(rows) and np.array_equal(tok, atok[rows]) and np.array_equal(o, ao) and torch.equal(kv, akv)
    assert np.allclose(conf, aconf[rows], rtol=1.3e-4, atol=0)       # as above: the chunks of the two runs differ in length
