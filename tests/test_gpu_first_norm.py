"""The first kernel of a forward: row tables and embeddings of refreshes and steps.  The O and down projections are zero, so the
residual stream that odb_debug_read returns is the embedding row of the token that each row was given, bit for bit."""
import dataclasses

import numpy as np
import pytest
import torch

import synth
from gpu_common import engine, requires_gpu

SETS = [(), (1,), (2,), (1, 2), (3,), (1, 2, 3), (4,), (1, 2, 3, 4)]    # ranks that a copy fills
D = 1216                                                                  # two slices of columns, the second not full


def model(E, batch, max_seq, block):
    shape = dataclasses.replace(synth.TINY, n_layers=1, d_model=D, n_heads=19, d_ffn=64, vocab=500, mask_id=499, eos_id=498)
    g = torch.Generator(device="cuda").manual_seed(1)

    def rnd(*n):
        return torch.randn(*n, generator=g, device="cuda").to(torch.bfloat16)

    ones = torch.ones(D, device="cuda")
    t = {"embed": rnd(500, D), "final_norm": ones, "norm1": [ones], "norm2": [ones], "lm_head": None,
         "wqkv": [E.pack_weight(rnd(3 * D, D))], "wo": [E.pack_weight(torch.zeros(D, D, device="cuda", dtype=torch.bfloat16))],
         "wgu": [E.pack_gate_up(rnd(128, D))], "wd": [E.pack_weight(torch.zeros(D, 64, device="cuda", dtype=torch.bfloat16))]}
    return shape, t, E.Model(shape, t, max_batch=batch, max_seq=max_seq, max_block=block, max_copies=8, with_lm_head=False)


@requires_gpu
@pytest.mark.parametrize("batch,away,block,copies,decoded", [
    (1, (), 1, 1, 0),              # one row
    (1, (), 64, 8, 40),            # the decoded-share layout, positions in both words of the mask; 64 + 7 * 24 rows
    (3, (1,), 33, 4, 0),           # 2 * 132 rows: four to a block, a block across two sequences
    (5, (0, 4), 24, 8, 15),        # inactive ones in front and behind
    (64, (7, 8, 63), 5, 4, 2),     # the largest batch
])
def test_rows_and_embeddings(batch, away, block, copies, decoded):
    E = engine()
    lens = [(3 + 5 * i % 37, block + i % 11) for i in range(batch)]
    shape, t, gm = model(E, batch, max(p + n for p, n in lens), block)
    sess = E.Session(gm, poison=True)
    embed = t["embed"].float().cpu().numpy()
    rng = np.random.default_rng(3)
    ids = []
    for i, (p, n) in enumerate(lens):
        x = np.full(p + n, shape.mask_id, dtype=np.int32)
        x[:p] = rng.integers(0, 498, p)
        x[p + rng.permutation(block)[:decoded]] = 7 + i
        ids.append(x)
        sess.set_sequence(i, x, p)
    for i in away:
        sess.set_active(i, False)
    there = [i for i in range(batch) if i not in away]

    par = E.DecodeParams(block_len=block, n_copies=copies)
    sess.refresh_prefill(par, 0)
    assert np.array_equal(sess.debug_read("row_tok"), np.concatenate([ids[i] for i in there]))
    assert np.array_equal(sess.debug_read("row_pos"), np.concatenate([np.arange(len(ids[i])) for i in there]))
    assert np.array_equal(sess.debug_read("hidden"), embed[np.concatenate([ids[i] for i in there])])
    sess.unmask_accept(par, True)

    sess.block_decode_step(par)
    tok, pos, copy = [], [], []
    for i in there:
        p, x = lens[i][0], ids[i]
        masked = [q for q in range(p, p + block) if x[q] == shape.mask_id]
        share = copies == 8 and decoded >= (4 * block + 6) // 7
        ranks = min(len(masked), {1: 0, 4: 2, 8: 4}[copies])
        for c, s in enumerate(y for y in SETS[: 8 if share else min(copies, 4)] if all(r <= ranks for r in y)):
            for q in range(p, p + block):
                if share and c and q not in masked:
                    continue
                tok.append(0 if q in [masked[r - 1] for r in s] else x[q])
                pos.append(q)
                copy.append(c)
    for name, want in (("row_tok", tok), ("row_pos", pos), ("row_copy", copy)):
        assert np.array_equal(sess.debug_read(name), np.array(want)), name
    assert np.array_equal(sess.debug_read("hidden"), embed[tok])
    assert sess.status() == 0
    sess.unmask_accept(par, False)
    sess.close(); gm.close()
