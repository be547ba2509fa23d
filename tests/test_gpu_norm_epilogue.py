"""The norm in the epilogue of an unsplit projection of few rows (odb_api.cu: norm_fits): lockstep with the oracle around its limits, in
models with and without LM head (without, the down projection of up to twelve k-blocks takes it too)."""
import dataclasses

import numpy as np
import pytest
import torch

import synth
from gpu_common import engine, requires_gpu
from test_gpu_many_rows import HD64, test_refresh_of_many_rows as check_refresh


@requires_gpu
@pytest.mark.parametrize("heads,rows", [(1, 2), (2, 16), (3, 17), (4, 31), (4, 32), (4, 33), (7, 32), (8, 32)])   # d 64 .. 512, whole and part tiles
def test_refresh_with_lm_head(heads, rows):
    check_refresh(dataclasses.replace(HD64, n_heads=heads, d_model=64 * heads), rows - rows // 2, rows // 2)


@requires_gpu
@pytest.mark.parametrize("heads,ffn,rows", [(1, 64, 1), (4, 688, 16), (4, 768, 32), (4, 784, 32), (5, 704, 31), (16, 256, 32)])   # 1 to 13 k-blocks
def test_residual_stream_without_lm_head(heads, ffn, rows):
    """Against 64 bits: two layers, so that the norm behind each projection is used."""
    E = engine()
    d = 64 * heads
    shape = dataclasses.replace(synth.TINY, n_layers=2, d_model=d, n_heads=heads, d_ffn=ffn, vocab=64, mask_id=63, eos_id=62)
    g = torch.Generator().manual_seed(heads)

    def mat(*n):
        return (torch.randn(*n, generator=g) * 1.28 / n[-1] ** 0.5).to(torch.bfloat16).cuda()

    def gain():
        return (1 + 0.1 * torch.randn(d, generator=g)).cuda()

    w = {"embed": mat(64, d), "norm1": [gain(), gain()], "norm2": [gain(), gain()], "wqkv": [mat(3 * d, d), mat(3 * d, d)],
         "wo": [mat(d, d), mat(d, d)], "wgu": [mat(2 * ffn, d), mat(2 * ffn, d)], "wd": [mat(d, ffn), mat(d, ffn)]}
    t = {"embed": w["embed"], "final_norm": gain(), "norm1": w["norm1"], "norm2": w["norm2"], "lm_head": None,
         "wgu": [E.pack_gate_up(x) for x in w["wgu"]], **{k: [E.pack_weight(x) for x in w[k]] for k in ("wqkv", "wo", "wd")}}
    gm = E.Model(shape, t, max_batch=1, max_seq=max(rows, 2), max_block=1, max_copies=1, with_lm_head=False)
    sess = E.Session(gm, poison=True)
    ids = np.random.default_rng(rows).integers(0, 62, rows).astype(np.int32)
    ids[-1] = 63
    sess.set_sequence(0, ids, rows - 1)
    sess.refresh_prefill(E.DecodeParams(block_len=1), 0)
    got = torch.from_numpy(sess.debug_read("hidden")).double()
    assert sess.status() == 0

    def norm(x, k):
        return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + shape.rms_eps) * k.double().cpu()

    h = w["embed"].double().cpu()[torch.from_numpy(ids).long()]
    pos = torch.arange(rows, dtype=torch.float64)[:, None]
    ang = pos * shape.rope_theta ** (-2.0 * torch.arange(32, dtype=torch.float64) / 64)
    c, s = ang.cos()[:, None], ang.sin()[:, None]
    for l in range(2):
        q, k, v = ((norm(h, w["norm1"][l]) @ w["wqkv"][l].double().cpu().T).view(rows, 3, heads, 64).unbind(1))
        q, k = (torch.cat([x[..., :32] * c - x[..., 32:] * s, x[..., 32:] * c + x[..., :32] * s], -1) for x in (q, k))
        o = torch.einsum("hqk,khd->qhd", torch.softmax(torch.einsum("qhd,khd->hqk", q, k) / 8, -1), v).reshape(rows, d)
        h = h + o @ w["wo"][l].double().cpu().T
        up = norm(h, w["norm2"][l]) @ w["wgu"][l].double().cpu().T
        h = h + (torch.nn.functional.silu(up[:, :ffn]) * up[:, ffn:]) @ w["wd"][l].double().cpu().T
    # eight bf16 roundings a layer (operands of four projections, q, k, v, P), each 2^-9 of the value at most and passed on with a gain of
    # about one: their sum, were they all to point the same way (they do not: 1e-2 is seen).  A row or tile gone wrong is off by 1.
    assert ((got - h).norm() / h.norm()).item() < 16 * 2.0 ** -9
    assert (got - h).abs().max().item() < 0.1 * h.pow(2).mean().sqrt().item()
    sess.close(); gm.close()
