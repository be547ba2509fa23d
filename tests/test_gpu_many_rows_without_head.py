"""Refreshes of more than 128 rows in models without LM head, whose projections take K splits of their own (gemm_rows_splits) and an
unsplit QKV: the residual stream of two layers with real weights against 64 bits, at sizes that reach each of the split counts."""
import ctypes
import dataclasses

import numpy as np
import pytest
import torch

import synth
from gpu_common import engine, requires_gpu


def exact(shape, w, ids):
    """The residual stream of one sequence in 64 bits, on the device."""
    n, hd, heads, ffn, half = len(ids), shape.head_dim, shape.n_heads, shape.d_ffn, shape.head_dim // 2

    def norm(x, gain):
        return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + shape.rms_eps) * gain.double()

    h = w["embed"].double()[torch.from_numpy(ids).long().cuda()]
    freq = shape.rope_theta ** (-2.0 * torch.arange(half, dtype=torch.float64, device="cuda") / hd)
    ang = torch.arange(n, dtype=torch.float64, device="cuda")[:, None] * freq
    c, s = ang.cos()[:, None], ang.sin()[:, None]
    for l in range(shape.n_layers):
        q, k, v = (norm(h, w["norm1"][l]) @ w["wqkv"][l].double().T).view(n, 3, heads, hd).unbind(1)
        q, k = (torch.cat([x[..., :half] * c - x[..., half:] * s, x[..., half:] * c + x[..., :half] * s], -1) for x in (q, k))
        p = torch.softmax(torch.einsum("qhd,khd->hqk", q, k) / hd ** 0.5, -1)
        h = h + torch.einsum("hqk,khd->qhd", p, v).reshape(n, -1) @ w["wo"][l].double().T
        up = norm(h, w["norm2"][l]) @ w["wgu"][l].double().T
        h = h + (torch.nn.functional.silu(up[:, :ffn]) * up[:, ffn:]) @ w["wd"][l].double().T
    return h


@requires_gpu
@pytest.mark.parametrize("hd,heads,ffn,lens,splits", [
    (64, 4, 736, [200], (1, 1)),               # added to the residual stream in the epilogue
    (64, 4, 1472, [130], (1, 2)),
    (64, 4, 8192, [200], (1, 16)),             # as many as the norm adds up
    (128, 4, 4096, [257], (1, 8)),             # one row in the second row tile
    (64, 16, 2816, [300], (2, 4)),             # four rows to a block of the norm behind, up to four partials
    (128, 8, 5504, [400], (2, 9)),             # more: one row to a block
    (64, 16, 2816, [581, 17, 519], (2, 3)),    # a ragged batch
    (128, 16, 5504, [300, 213], (3, 3)),
    (64, 16, 1472, [1500], (1, 2)),
    (128, 3, 736, [150, 101], None),           # three weight tiles: not the many-row kernel
])
def test_residual_stream(hd, heads, ffn, lens, splits):
    E = engine()
    from paper_2511_21759_b200 import binding as B
    d, rows = hd * heads, sum(lens)
    rule = B.lib()._ZN3odb16gemm_rows_splitsEiii
    rule.argtypes, rule.restype = (ctypes.c_int,) * 3, ctypes.c_int
    assert splits is None or (rule(rows, d, d), rule(rows, d, ffn)) == splits
    shape = dataclasses.replace(synth.TINY, n_layers=2, d_model=d, n_heads=heads, head_dim=hd, d_ffn=ffn, vocab=64, mask_id=63, eos_id=62)
    g = torch.Generator(device="cuda").manual_seed(d + ffn)

    def mat(*n):
        return (torch.randn(*n, generator=g, device="cuda") * 1.28 / n[-1] ** 0.5).to(torch.bfloat16)

    def gain():
        return 1 + 0.1 * torch.randn(d, generator=g, device="cuda")

    w = {"embed": mat(64, d)}
    for k, n in (("norm1", None), ("norm2", None), ("wqkv", (3 * d, d)), ("wo", (d, d)), ("wgu", (2 * ffn, d)), ("wd", (d, ffn))):
        w[k] = [mat(*n) if n else gain() for _ in range(2)]
    t = {"embed": w["embed"], "final_norm": gain(), "norm1": w["norm1"], "norm2": w["norm2"], "lm_head": None,
         "wgu": [E.pack_gate_up(x) for x in w["wgu"]], **{k: [E.pack_weight(x) for x in w[k]] for k in ("wqkv", "wo", "wd")}}
    gm = E.Model(shape, t, max_batch=len(lens), max_seq=max(lens), max_block=1, max_copies=1, with_lm_head=False)
    sess = E.Session(gm, poison=True)
    ids = []
    for i, n in enumerate(lens):
        x = np.random.default_rng(i).integers(0, 62, n).astype(np.int32)
        x[-1] = 63
        ids.append(x)
        sess.set_sequence(i, x, n - 1)
    sess.refresh_prefill(E.DecodeParams(block_len=1), 0)
    got = torch.from_numpy(sess.debug_read("hidden")).cuda().double()
    assert sess.status() == 0 and len(got) == rows
    want = torch.cat([exact(shape, w, x) for x in ids])
    # as in the few-row test: eight bf16 roundings a layer, 2^-9 of the value each, were they all to point the same way.  A split left
    # out or counted twice, or a row or tile gone wrong, is off by a third or more of the projection's part of the stream.
    row_error = (got - want).norm(dim=1) / want.norm(dim=1)
    assert row_error.max().item() < 16 * 2.0 ** -9
    assert (got - want).abs().max().item() < 0.1 * want.pow(2).mean().sqrt().item()
    sess.close(); gm.close()
