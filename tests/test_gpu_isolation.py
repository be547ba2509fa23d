"""A sequence whose rows are not finite leaves the others of its batch, and the next occupant of its slot, alone: their results are
the bits they have without it.  Rows of tiles behind a sequence's last key are other sequences', or left over in the cache."""
import dataclasses

import numpy as np
import pytest

import synth
from gpu_common import engine, requires_gpu
from test_gpu_many_rows import HD64, HD128

NAN_ID = 9          # its embedding is not finite


def shape_of(hd, heads):
    return dataclasses.replace(HD64 if hd == 64 else HD128, n_layers=2, n_heads=heads, d_model=hd * heads, d_ffn=256)


def model(E, shape, head, **kw):
    gm = E.Model.from_synth(shape, seed=5, with_lm_head=head, **kw)
    t = dict(gm.t)
    t["embed"] = t["embed"].clone()
    t["embed"][NAN_ID] = float("nan")
    gm.close()
    return E.Model(shape, t, with_lm_head=head, **kw)


def ids(i, p, n, shape):
    x = synth.sequence(5, i, p, n, shape)
    x[x == NAN_ID] += 1
    return x


def forward(sess, par):
    """The residual stream of a refresh and of a step, by sequence."""
    out = []
    for step in (False, True):
        sess.block_decode_step(par) if step else sess.refresh_prefill(par, 0)
        hidden = sess.debug_read("hidden")
        seq = np.cumsum(np.r_[1, starts(sess.debug_read("row_pos"), sess.debug_read("row_copy"))]) - 1
        out.append([hidden[seq == i] for i in range(seq[-1] + 1)])
        sess.unmask_accept(par, not step)
    assert sess.status() == 0
    return out


def starts(pos, copy):
    """Rows are in sequence order, copy 0 first: whether row r + 1 begins a sequence."""
    return (copy[1:] == 0) & ((copy[:-1] != 0) | (pos[1:] != pos[:-1] + 1))


@requires_gpu
@pytest.mark.parametrize("hd,heads,copies,block,batch", [
    (64, 32, 1, 24, 3),       # refresh on the tensor cores, the step on mma.sync
    (64, 32, 1, 24, 10),      # both on the tensor cores: one copy, a CTA per item
    (64, 32, 4, 24, 1 + 1),   # several copies, key splits
    (128, 32, 4, 24, 2),
    (128, 32, 4, 32, 4),      # without
    (128, 32, 1, 20, 5),
    (128, 4, 8, 32, 2),       # few work items
])
def test_other_sequences_keep_their_bits(hd, heads, copies, block, batch):
    E = engine()
    shape = shape_of(hd, heads)
    lens = [(100 + 7 * i, 57 + 5 * (i % 3)) for i in range(batch)]
    kw = dict(max_batch=batch, max_seq=max(p + n for p, n in lens) + 70, max_block=block, max_copies=8)
    gm = model(E, shape, False, **kw)
    par = E.DecodeParams(block_len=block, n_copies=copies, alp=False)
    bad, got = 1, {}
    for nan in (False, True):
        sess = E.Session(gm, poison=True)
        for i, (p, n) in enumerate(lens):
            x = ids(i, p, n, shape)
            if nan and i == bad:
                x[:p] = NAN_ID
            sess.set_sequence(i, x, p)
        got[nan] = forward(sess, par)
        # the slot's next occupant is shorter: behind its last key the cache holds what was there before
        p, n = lens[bad]
        for i, (q, m) in enumerate(lens):
            q = p - 41 if i == bad else q
            sess.set_sequence(i, ids(i, q, m, shape), q)
        got["reused", nan] = forward(sess, par)
        sess.close()
    assert not np.isfinite(got[True][0][bad]).any()
    for clean, other in zip(got[False], got[True]):
        for i in range(batch):
            assert i == bad or (np.isfinite(clean[i]).all() and np.array_equal(clean[i], other[i])), i
    for clean, other in zip(got["reused", False], got["reused", True]):
        assert all(np.isfinite(a).all() and np.array_equal(a, b) for a, b in zip(clean, other))
    gm.close()


@requires_gpu
@pytest.mark.parametrize("copies,resident", [(1, False), (4, False), (4, True), (8, False)])
def test_a_row_without_a_greedy_token_counts_as_eos(copies, resident):
    """A NaN prompt: every response row's logits are NaN after a refresh.  What is committed stays inside the vocabulary and the block
    ends; the other sequences decode what they decode without it."""
    E = engine()
    shape = dataclasses.replace(HD128, n_heads=4, d_model=512, d_ffn=256)
    lens, block, bad = [(40, 32), (37, 32), (50, 24)], 16, 1
    gm = model(E, shape, True, max_batch=3, max_seq=80, max_block=block, max_copies=8)
    par = E.DecodeParams(block_len=block, n_copies=copies, alp=False)
    done = {}
    for nan in (False, True):
        sess = E.Session(gm, poison=True)
        for i, (p, n) in enumerate(lens):
            x = ids(i, p, n, shape)
            if nan and i == bad:
                x[:p] = NAN_ID
            sess.set_sequence(i, x, p)
        sess.refresh_prefill(par, 0)
        assert np.isnan(sess.debug_read("hidden")).any() == nan
        res = sess.unmask_accept(par, True)
        if nan:
            r = res[bad]
            assert [(r.accepted_pos[j], r.accepted_tok[j]) for j in range(r.n_accepted)] == [(37, shape.eos_id)]
        left = max(r.masks_left for r in res)
        for _ in range(block):
            if left == 0:
                break
            if resident:
                left = max(r.masks_left for r in sess.decode_block_resident(par, block)[-1])
            else:
                sess.block_decode_step(par)
                left = max(r.masks_left for r in sess.unmask_accept(par, False))
        assert left == 0 and sess.status() == 0
        done[nan] = [sess.get_tokens(i)[: p + block] for i, (p, n) in enumerate(lens)]
        sess.close()
    gm.close()
    assert ((done[True][bad] >= 0) & (done[True][bad] < shape.vocab) & (done[True][bad] != shape.mask_id)).all()
    for i in (0, 2):
        assert np.array_equal(done[False][i], done[True][i])
