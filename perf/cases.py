"""Workloads of the block-decoding library, as a program that serves a diffusion LLM meets them.

Every case goes through `engine.Model` / `engine.Session`, the calls a serving loop makes:

  step      one decoding iteration of the current block: block_decode_step, then unmask_accept
  resident  several iterations without returning to the host: decode_block_resident
  refresh   the cache refresh at a block boundary: refresh_prefill, then unmask_accept(after_refresh)
  request   a new request up to its first committed tokens: set_sequence for every sequence of the batch,
            refresh_prefill with the LM head, unmask_accept(after_refresh)

step, resident and refresh run on models built without LM head, whose accept commits nothing and lays out the same
step again, so that a pass can be repeated on one state; their result is the residual stream (and the K/V cache a
refresh writes).  request runs with the LM head; logits never exist in the product path, its result is the confidence
and greedy token of every response row and the K/V cache.

Shapes: the 8B-shaped layer (d 4096, 32 heads of 128, FFN 12288, vocabulary 126464) of the full-size workloads, the
tiny model (2 layers, d 256, 4 heads of 64, FFN 688) and two generic widths between them.  Weights are
N(0, 1.28 / sqrt(d)), which is N(0, 0.02) at d 4096; gains scatter around 1.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2511_21759_b200 import engine as E


@dataclasses.dataclass(frozen=True)
class Shape:
    n_layers: int
    d_model: int
    n_heads: int
    head_dim: int
    d_ffn: int
    vocab: int
    mask_id: int
    eos_id: int
    rope_theta: float = 500000.0
    rms_eps: float = 1e-5


_TINY = dict(d=256, heads=4, hd=64, ffn=688, vocab=2048)
_SMALL64 = dict(d=1024, heads=16, hd=64, ffn=2816, vocab=32000)
_MID128 = dict(d=2048, heads=16, hd=128, ffn=5504, vocab=32000)
_8B = dict(d=4096, heads=32, hd=128, ffn=12288, vocab=126464)


def _case(name, kind, size, layers=1, batch=1, prompt=256, gen=256, block=32, copies=1, decoded=0, ragged=0, iters=0):
    c = dict(kind=kind, layers=layers, batch=batch, prompt=prompt, gen=gen, block=block, copies=copies, decoded=decoded,
             ragged=ragged, iters=iters, **size)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the tiny model one block iteration at a time: launches and host calls are the whole cost
        _case("tiny_step", "step", _TINY, layers=2, prompt=64, gen=64, block=16),
        # the plain decode step at batch 1, one layer of the 8B shape: a read of the weights
        _case("layer_step", "step", _8B, prompt=256, gen=256),
        # the same with the four speculative copies, 128 query rows
        _case("layer_step_4_copies", "step", _8B, prompt=512, gen=512, copies=4),
        # eight copies in the decoded-share layout late in a block, odd lengths: 24 + 7 * 9 rows
        _case("layer_step_decoded_share", "step", _8B, prompt=331, gen=205, block=24, copies=8, decoded=15),
        # a small batch of unequal requests without speculation
        _case("layer_step_batch4", "step", _8B, batch=4, prompt=417, gen=256, ragged=29),
        # a serving batch with speculation: 16 sequences of unequal length, blocks of 64, 4096 query rows
        _case("layer_step_batch16", "step", _8B, batch=16, prompt=1024, gen=1024, block=64, copies=4, ragged=57),
        # the decode loop of a block as a latency-minded server runs it, four layers deep
        _case("resident_loop", "resident", _8B, layers=4, prompt=512, gen=256, iters=8),
        # the block-boundary refresh of one request
        _case("layer_refresh", "refresh", _8B, prompt=512, gen=256),
        # ... and of the serving batch, the largest call
        _case("layer_refresh_batch16", "refresh", _8B, batch=16, prompt=1024, gen=1024, block=64, ragged=57),
        # head dimension 64 and a middling width, two requests
        _case("small_refresh_hd64", "refresh", _SMALL64, layers=2, batch=2, prompt=389, gen=192, ragged=41),
        # a short request: every row is a response row or nearly, the LM head is most of the work
        _case("short_request", "request", _8B, prompt=17, gen=31),
        # a whole request: four layers, LM head and confidence over the whole response
        _case("request", "request", _8B, layers=4, prompt=512, gen=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "resident", "refresh", "refresh", "request"])
    size = rng.choice([_TINY, _SMALL64, _MID128, _8B, _8B, _8B])
    batch = _log_int(rng, 1, 4 if kind == "request" else 16)
    prompt, gen = _log_int(rng, 16, 900), _log_int(rng, 32, 900)
    block = min(rng.choice([8, 16, 24, 32, 32, 37, 48, 64]), gen)
    copies = rng.choice([1, 1, 4, 4, 8]) if kind in ("step", "resident") else 1
    decoded = rng.randrange(0, block - 4) if kind in ("step", "resident") else 0
    layers = rng.choice([1, 2]) if batch * (prompt + gen) < 4000 else 1
    iters = rng.randrange(2, 9) if kind == "resident" else 0
    ragged = rng.randrange(0, 40) if batch > 1 else 0
    return _case(None, kind, size, layers, batch, prompt, gen, block, copies, decoded, ragged, iters)


# ------------------------------------------------------------------------------------------------- inputs

def _lengths(case):
    """Prompt and response length of every sequence: unequal when `ragged`, never shorter than a block."""
    return [(max(1, case["prompt"] - 3 * i if case["ragged"] else case["prompt"]),
             max(case["block"], case["gen"] - case["ragged"] * i)) for i in range(case["batch"])]


def _shape(case):
    return Shape(case["layers"], case["d"], case["heads"], case["hd"], case["ffn"], case["vocab"], case["vocab"] - 1,
                 case["vocab"] - 2)


def _weights(case, seed):
    """Row-major weights, the way a checkpoint holds them."""
    g = torch.Generator(device="cuda").manual_seed(2 * seed + 1)
    d, f, n = case["d"], case["ffn"], case["layers"]

    def mat(rows, cols, std):
        return torch.randn(rows, cols, generator=g, device="cuda", dtype=torch.bfloat16).mul_(std)

    def gain():
        return 1.0 + 0.1 * torch.randn(d, generator=g, device="cuda", dtype=torch.float32)

    std = 1.28 / math.sqrt(d)
    w = {"embed": mat(case["vocab"], d, 0.02), "final_norm": gain(), "norm1": [], "norm2": [], "wqkv": [], "wo": [],
         "wgu": [], "wd": [], "lm_head": None}
    for _ in range(n):
        w["norm1"].append(gain())
        w["norm2"].append(gain())
        w["wqkv"].append(mat(3 * d, d, std))
        w["wo"].append(mat(d, d, std))
        w["wgu"].append(mat(2 * f, d, std))
        w["wd"].append(mat(d, f, std))
    if case["kind"] == "request":
        w["lm_head"] = mat(case["vocab"], d, std)
    return w


def _ids(case, seed):
    """Token ids per sequence: a random prompt, then masks, of which `decoded` in the first block are already filled."""
    rng = np.random.default_rng(seed)
    mask = case["vocab"] - 1
    out = []
    for p, n in _lengths(case):
        x = np.full(p + n, mask, dtype=np.int32)
        x[:p] = rng.integers(0, case["vocab"] - 2, p)
        at = rng.permutation(case["block"])[: case["decoded"]]
        x[p + at] = rng.integers(0, case["vocab"] - 2, len(at))
        out.append(x)
    return out


class _State:
    def __init__(self, model, sess):
        self.model, self.sess = model, sess

    def __del__(self):
        self.sess.close()
        self.model.close()


def _in_workspace(sess, what):
    """The buffer that debug_read(what) copies from, as a view of the caller-owned workspace: a program that goes on
    with the values on the device reads them in place.  Found by its contents."""
    ref = sess.debug_read(what)
    words = sess.ws[: sess.ws.numel() // 4 * 4].view(torch.int32)
    flat = torch.from_numpy(np.ascontiguousarray(ref).view(np.int32).reshape(-1)).to(words.device)
    n = flat.numel()
    at = []
    for lo in range(0, words.numel() - n + 1, 1 << 28):
        part = words[lo: min(lo + (1 << 28), words.numel() - n + 1)]
        at += (torch.nonzero(part == flat[0]).reshape(-1) + lo).tolist()
    at = [a for a in at if a % 64 == 0 and bool((words[a: a + n] == flat).all())]
    assert len(at) == 1, f"{what}: {len(at)} places"
    return words[at[0]: at[0] + n].view(torch.float32 if ref.dtype == np.float32 else torch.int32).view(ref.shape)


def prepare(case, seed):
    w = _weights(case, seed)
    head = case["kind"] == "request"
    t = {"embed": w["embed"], "final_norm": w["final_norm"], "norm1": w["norm1"], "norm2": w["norm2"],
         "lm_head": E.pack_weight(w["lm_head"]) if head else None}
    for k in ("wqkv", "wo", "wd"):
        t[k] = [E.pack_weight(x) for x in w[k]]
    t["wgu"] = [E.pack_gate_up(x) for x in w["wgu"]]
    del w
    model = E.Model(_shape(case), t, max_batch=case["batch"], max_seq=max(p + n for p, n in _lengths(case)),
                    max_block=case["block"], max_copies=case["copies"], with_lm_head=head)
    sess = E.Session(model)
    s = _State(model, sess)
    s.kind, s.iters = case["kind"], case["iters"]
    s.params = E.DecodeParams(block_len=case["block"], n_copies=case["copies"])
    s.ids, s.prompts = _ids(case, seed), [p for p, _ in _lengths(case)]
    for i, x in enumerate(s.ids):
        sess.set_sequence(i, x, s.prompts[i])
    sess.refresh_prefill(s.params, 0)
    if head:
        s.conf, s.tok = _in_workspace(sess, "conf"), _in_workspace(sess, "tok")
    else:
        s.hidden = _in_workspace(sess, "hidden")
    sess.unmask_accept(s.params, True)
    if s.kind in ("step", "resident"):
        sess.block_decode_step(s.params)
        rows = len(sess.debug_read("row_pos"))
        sess.unmask_accept(s.params, False)
        flat = s.hidden.reshape(-1)
        s.hidden = flat.as_strided((rows, case["d"]), (case["d"], 1), flat.storage_offset())
    s.kv = sess.kv.view(torch.bfloat16).view(case["batch"], case["layers"], 2, case["heads"], -1, case["hd"])
    return s


def run(s):
    sess = s.sess
    if s.kind == "step":
        sess.block_decode_step(s.params)
        sess.unmask_accept(s.params, False)
        return s.hidden
    if s.kind == "resident":
        sess.decode_block_resident(s.params, s.iters)
        return s.hidden
    if s.kind == "request":
        for i, x in enumerate(s.ids):
            sess.set_sequence(i, x, s.prompts[i])
    sess.refresh_prefill(s.params, 0)
    sess.unmask_accept(s.params, True)
    return (s.conf, s.tok, s.kv) if s.kind == "request" else (s.hidden, s.kv)


# ------------------------------------------------------------------------------------------------- size and error

def _copies(case):
    """Rank subsets of the copies of a step, and whether it is in the decoded-share layout."""
    left = case["block"] - case["decoded"]
    ranks = min(left, {1: 0, 4: 2, 8: 4}[case["copies"]])
    shared = case["copies"] == 8 and case["decoded"] >= (4 * case["block"] + 6) // 7
    sets = [(), (1,), (2,), (1, 2), (3,), (1, 2, 3), (4,), (1, 2, 3, 4)]
    sets = sets[: 8 if shared else min(case["copies"], 4)]
    return [y for y in sets if all(r <= ranks for r in y)], shared


def _step_rows(case):
    sets, shared = _copies(case)
    return case["block"] + (len(sets) - 1) * (case["block"] - case["decoded"] if shared else case["block"])


def work(case):
    d, f, n = case["d"], case["ffn"], case["layers"]
    layer = 4 * d * d + 3 * f * d
    lens = [p + g for p, g in _lengths(case)]
    if case["kind"] in ("step", "resident"):
        m = _step_rows(case)
        rows = m * len(lens)
        ctx = sum(t - case["block"] for t in lens)
        one_b = n * (2 * layer + 4 * d * ctx) + 6 * d * rows
        one_f = n * (2 * layer * rows + 4 * d * m * (ctx + case["block"] * len(lens)))
        times = max(1, case["iters"])
        return {"bytes": times * one_b, "flops": times * one_f}
    rows = sum(lens)
    b = n * (2 * layer + 4 * d * rows) + 2 * d * rows
    fl = n * (2 * layer * rows + 4 * d * sum(t * t for t in lens))
    if case["kind"] == "request":
        gen = sum(g for _, g in _lengths(case))
        # the last layer's output projection and FFN are needed for response rows only
        fl -= 2 * (layer - 3 * d * d) * (rows - gen) + 4 * d * sum(p * (p + g) for p, g in _lengths(case))
        b += 2 * d * case["vocab"] + 8 * gen
        fl += 2 * d * case["vocab"] * gen
    else:
        b += 4 * d * rows
    return {"bytes": b, "flops": fl}


def tolerance(case):
    # About four times what the same forward shows with its sums split in other places (other K splits, single CTAs
    # instead of pairs, the other attention kernel): 2.3e-3 per layer in the residual stream, 1.5e-2 of the rms at
    # worst; through the LM head 5.6e-3 in the confidences after one layer and 6.9e-3 after four, 6 % of the greedy
    # tokens (a vocabulary of 126464 random logits: the two best often lie closer than the logits' error).
    n = case["layers"]
    if case["kind"] == "request":
        return {"rel": 2.2e-2 * n ** 0.25, "max": 0.1, "differ": 0.25}
    return {"rel": 1e-2 * math.sqrt(n), "max": 6e-2 * math.sqrt(n)}


# ------------------------------------------------------------------------------------------------- 64-bit reference

def _norm(x, gain, eps):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + eps) * gain.double()


def _rope(x, pos, theta):
    """x [rows][heads][hd], rotating pairs (i, i + hd/2)."""
    half = x.shape[-1] // 2
    inv = torch.tensor(theta, dtype=torch.float64) ** (-2.0 * torch.arange(half, dtype=torch.float64) / x.shape[-1])
    ang = pos.double()[:, None] * inv.to(x.device)[None, :]
    c, s = ang.cos()[:, None, :], ang.sin()[:, None, :]
    a, b = x[..., :half], x[..., half:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


def _attend(q, k, v, visible=None):
    """q [rows][heads][hd] over k, v [keys][heads][hd]."""
    s = torch.einsum("qhd,khd->hqk", q, k) / math.sqrt(q.shape[-1])
    if visible is not None:
        s = s.masked_fill(~visible[None], -math.inf)
    return torch.einsum("hqk,khd->qhd", torch.softmax(s, -1), v).reshape(q.shape[0], -1)


def _layer(case, w, l, h, pos, keys):
    """One layer over the rows h; keys(q, k, v) is the attention.  Returns h, k, v."""
    d, f, shape = case["d"], case["ffn"], _shape(case)
    heads = (-1, case["heads"], case["hd"])
    qkv = _norm(h, w["norm1"][l], shape.rms_eps) @ w["wqkv"][l].double().T
    q, k = (_rope(qkv[:, i * d:(i + 1) * d].reshape(heads), pos, shape.rope_theta) for i in (0, 1))
    v = qkv[:, 2 * d:].reshape(heads)
    h = h + keys(q, k, v) @ w["wo"][l].double().T
    up = _norm(h, w["norm2"][l], shape.rms_eps) @ w["wgu"][l].double().T
    return h + (torch.nn.functional.silu(up[:, :f]) * up[:, f:]) @ w["wd"][l].double().T, k, v


def exact(case, seed):
    with torch.no_grad():
        w, ids = _weights(case, seed), [torch.from_numpy(x).long().cuda() for x in _ids(case, seed)]
        hidden, caches = [], []
        for x in ids:
            h, pos, cache = w["embed"][x].double(), torch.arange(len(x), device="cuda"), []
            for l in range(case["layers"]):
                h, k, v = _layer(case, w, l, h, pos, _attend)
                cache.append((k, v))
            hidden.append(h)
            caches.append(cache)
        if case["kind"] in ("step", "resident"):
            return torch.cat([_exact_step(case, w, x, p, c) for x, (p, _), c in zip(ids, _lengths(case), caches)])
        longest = max(len(x) for x in ids)
        kv = torch.zeros(case["batch"], case["layers"], 2, case["heads"], longest, case["hd"], dtype=torch.float64,
                         device="cuda")
        for i, cache in enumerate(caches):
            for l, pair in enumerate(cache):
                for j in (0, 1):
                    kv[i, l, j, :, : len(ids[i])] = pair[j].transpose(0, 1)
        if case["kind"] == "refresh":
            return torch.cat(hidden), kv
        conf, tok = [], []
        for h, (p, _) in zip(hidden, _lengths(case)):
            logits = _norm(h[p:], w["final_norm"], _shape(case).rms_eps) @ w["lm_head"].double().T
            logits[:, case["vocab"] - 1] = -math.inf
            best = torch.softmax(logits, -1).max(-1)
            conf.append(best.values)
            tok.append(best.indices.int())
        return torch.cat(conf), torch.cat(tok), kv


def _exact_step(case, w, x, start, cache):
    """The rows of one sequence's step: copy 0 holds the block, copy c fills the first masked positions of its rank set
    with token 0; in the decoded-share layout a copy holds the masked positions only and sees copy 0's decoded ones."""
    sets, shared = _copies(case)
    end, mask = start + case["block"], case["vocab"] - 1
    masked = [p for p in range(start, end) if int(x[p]) == mask]
    copy, pos, tok = [], [], []
    for c, ranks in enumerate(sets):
        fills = {masked[r - 1] for r in ranks}
        for p in range(start, end):
            if shared and c and p not in masked:
                continue
            copy.append(c)
            pos.append(p)
            tok.append(0 if p in fills else int(x[p]))
    copy, pos, tok = (torch.tensor(t, device="cuda") for t in (copy, pos, tok))
    own = copy[:, None] == copy[None, :]
    if shared:
        own |= (copy == 0)[None, :] & (x[pos] != mask)[None, :]
    outside = torch.cat([torch.arange(0, start, device="cuda"), torch.arange(end, len(x), device="cuda")])
    visible = torch.cat([torch.ones(len(pos), len(outside), dtype=torch.bool, device="cuda"), own], 1)
    h = w["embed"][tok].double()
    for l in range(case["layers"]):
        ck, cv = (t[outside] for t in cache[l])
        h, _, _ = _layer(case, w, l, h, pos,
                         lambda q, k, v: _attend(q, torch.cat([ck, k]), torch.cat([cv, v]), visible))
    return h
