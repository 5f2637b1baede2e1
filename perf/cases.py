"""The calls a program makes of this library, as timed cases.

`listed()` are the fixed ones, `draw(rng)` gives more of the same ranges.  A case is a dict of plain
values; `prepare` makes what a program has in hand before the call (weights, contexts, inputs on the
GPU), `run` is one pass through the public entry points, `work` the bytes and operations of a pass,
`exact` the same outputs in 64 bits from plain torch and `tolerance` what another implementation of the
same precision would differ by.

Kinds
  reject    spd_reject_sample: the rejection rule alone on given probability rows -- the smallest call
            of a serving loop that has its own models (B = 1) up to a batch of 32 sequences.
  truncate  spd_truncate_probs: top-k / top-p rows in front of that rule.
  skinny    spd_skinny_gemm / spd_skinny_gemm_noalloc: one linear map on M <= 8 rows, bf16 and fp32.
  adapter   spd_image_adapter: the image projector in front of the target, 576 rows per image.
  prefill   spd_prefill: image rows + prompt through target and draft (time to the first token).
  draft     spd_draft: gamma tokens of the 115M draft, one after the other.
  verify    spd_verify: one target call on gamma + 1 rows against the cache and the rule.
  tree      spd_draft_tree + spd_verify_tree.
  batch     spd_batch_draft + spd_batch_verify: several sequences through one pass over the weights.
  generate  spd_generate of the small fp32 models: the latency floor of the whole block loop.

Target layers have the shapes of the LLaVA-7B-shaped workload (d 4096, 32 heads, ffn 11008, vocab
32000); the number of layers is small because every layer costs the same and a layer's weights alone
are larger than the L2 cache.  Drafts are the 115M shape and the one of the paper's Table 1.

Weights: matrices N(0, 0.02^2), the two that write the residual stream and the embedding scaled so that a
model's distributions are peaked on one token, as a trained model's mostly are.  Tokens are then the
same for any implementation of the same precision, and blocks are accepted in part or whole.
"""
from __future__ import annotations

import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2404_08856_b200 as spd

DEV = "cuda"
VOCAB = 32000
EPS, THETA = 1e-5, 10000.0


# ------------------------------------------------------------------------------------ models


def _cfg(layers, d, heads, ffn, vocab, tied, dtype):
    return SimpleNamespace(n_layers=layers, d_model=d, n_heads=heads, d_ffn=ffn, vocab=vocab, tied_embeddings=tied,
                           rms_eps=EPS, rope_theta=THETA, dtype=dtype)


def _models(case):
    """(target, draft) configurations of a case."""
    if case["target"] == "tiny":
        return _cfg(2, 256, 4, 688, 1024, False, "fp32"), _cfg(1, 128, 2, 344, 1024, False, "fp32")
    target = _cfg(case["layers"], 4096, 32, 11008, VOCAB, False, "bf16")
    if case["draft"] == "table1":
        return target, _cfg(4, 1024, 8, 2816, VOCAB, False, "bf16")
    return target, _cfg(12, 768, 12, 2048, VOCAB, True, "bf16")


def _weights(cfg, seed):
    """name -> tensor or list of tensors, on the GPU, in the model's type."""
    g = torch.Generator(DEV).manual_seed(seed)
    dt = torch.bfloat16 if cfg.dtype == "bf16" else torch.float32
    d, f = cfg.d_model, cfg.d_ffn
    # rows of the residual stream: the embedding stays the largest part of it, so that the LM head
    # (the embedding's own values) singles one token out
    e_std = max(0.02, 23.0 / math.sqrt(d) * 0.036)
    o_std = 0.25 * e_std / math.sqrt(2 * cfg.n_layers) / math.sqrt(f)

    def mat(rows, cols, std):
        return (torch.randn(rows, cols, generator=g, device=DEV) * std).to(dt)

    w = {"tok_embed": mat(cfg.vocab, d, e_std)}
    w["lm_head"] = w["tok_embed"]
    shapes = {"wq": (d, d, 0.02), "wk": (d, d, 0.02), "wv": (d, d, 0.02), "wo": (d, d, 2 * o_std),
              "w_gate": (f, d, 0.02), "w_up": (f, d, 0.02), "w_down": (d, f, 2 * o_std)}
    for name, shape in shapes.items():
        w[name] = [mat(*shape) for _ in range(cfg.n_layers)]
    ones = torch.ones(d, device=DEV)
    w["attn_norm"] = w["ffn_norm"] = [ones] * cfg.n_layers
    w["final_norm"] = ones
    return w


WEIGHT_SEED = 1          # one set of weights; the inputs come from the case's seed


def _context(case, max_seq, gamma_max):
    tc, dc = _models(case)
    return spd.Spd(tc, dc, _weights(tc, WEIGHT_SEED), _weights(dc, WEIGHT_SEED + 1), max_seq, gamma_max, 1.0,
                   bool(case["greedy"]), top_k=case.get("top_k", 0), top_p=case.get("top_p", 0.0))


def _rng(seed):
    return np.random.Generator(np.random.Philox(key=int(seed)))


def _uniforms(g, *shape):
    return (g.integers(0, 1 << 24, size=shape) / float(1 << 24)).astype(np.float32)


def _sequence(case, seed, index=0):
    """One sequence's inputs: image rows [m, d] (or None), prompt ids, the uniform of the first token."""
    tc, _ = _models(case)
    g = _rng(seed * 64 + index)
    image = None
    if case["image"]:
        t = torch.Generator(DEV).manual_seed(seed * 64 + index + 7)
        image = torch.randn(case["image"], tc.d_model, generator=t, device=DEV) * 0.02
    ids = g.integers(0, tc.vocab, size=case["prompt"]).astype(np.int32)
    return image, ids, float(_uniforms(g, 1)[0]), g


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _logits(ctx, out):
    ctx._check(spd.lib().spd_get_logits(ctx._ctx, _ptr(out), int(out.shape[0])))
    return out


# ------------------------------------------------------------------------------------ the same in 64 bits


class _Model64:
    """A decoder in 64 bits over whole rows (no cache)."""

    def __init__(self, cfg, seed):
        self.cfg, self.w = cfg, _weights(cfg, seed)

    def embed(self, ids):
        return self.w["tok_embed"][torch.as_tensor(np.asarray(ids, dtype=np.int64), device=DEV)].double()

    def logits(self, x, last):
        """Rows x [R, d] at positions 0..R-1; the logits of the last `last` rows."""
        c, w = self.cfg, self.w
        R, H, dh = x.shape[0], c.n_heads, c.d_model // c.n_heads
        inv = THETA ** (-torch.arange(0, dh, 2, device=DEV, dtype=torch.float64) / dh)
        ang = torch.arange(R, device=DEV, dtype=torch.float64)[:, None] * inv
        cos, sin = ang.cos()[None], ang.sin()[None]

        def norm(v, gain):
            return v / (v.square().mean(-1, keepdim=True) + EPS).sqrt() * gain.double()

        def rot(v):
            a, b = v[..., : dh // 2], v[..., dh // 2:]
            return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)

        hidden = torch.ones(R, R, dtype=torch.bool, device=DEV).triu(1)
        for l in range(c.n_layers):
            h = norm(x, w["attn_norm"][l])
            q, k, v = ((h @ w[n][l].double().T).view(R, H, dh).transpose(0, 1) for n in ("wq", "wk", "wv"))
            q, k = rot(q), rot(k)
            o = torch.empty_like(q)
            for i in range(0, H, 8):   # a few heads at a time: the score matrices are large
                s = (q[i:i + 8] @ k[i:i + 8].transpose(1, 2) / math.sqrt(dh)).masked_fill_(hidden, -math.inf)
                o[i:i + 8] = torch.softmax(s, -1) @ v[i:i + 8]
            x = x + o.transpose(0, 1).reshape(R, -1) @ w["wo"][l].double().T
            h = norm(x, w["ffn_norm"][l])
            a = torch.nn.functional.silu(h @ w["w_gate"][l].double().T) * (h @ w["w_up"][l].double().T)
            x = x + a @ w["w_down"][l].double().T
        return norm(x[R - last:], w["final_norm"]) @ w["lm_head"].double().T


def _pick64(p, u):
    """The token a uniform draws from a probability row."""
    return int(min(int((p.cumsum(0) <= u * p.sum()).sum()), p.numel() - 1))


def _truncate64(p, top_k, top_p):
    """top-k, then top-p, on one row: kept values over the kept mass."""
    mass = (p.to(torch.float64) * 2.0 ** 32).floor()
    order = torch.sort(p, descending=True, stable=True)[1]
    if 1 <= top_k < p.numel():
        order = order[:top_k]
    if top_p < 1.0:
        m = mass[order]
        p24 = math.floor(float(np.float32(top_p) * np.float32(2 ** 24)))
        need = max(1, -(-int(m.sum()) * p24 // 2 ** 24))
        order = order[: int((m.cumsum(0) < need).sum()) + 1]
    out = torch.zeros(p.numel(), dtype=torch.float64, device=p.device)
    out[order] = p[order].double() / (mass[order].sum() / 2.0 ** 32)
    return out


def _probs64(case, logits):
    p = torch.softmax(logits, -1)
    if not case["greedy"] and (case.get("top_k", 0) or 0 < case.get("top_p", 0.0) < 1):
        p = torch.stack([_truncate64(r.float(), case.get("top_k", 0), case.get("top_p") or 1.0) for r in p])
    return p


def _token64(case, row, u):
    return int(row.argmax()) if case["greedy"] else _pick64(_probs64(case, row[None])[0], u)


def _prompt64(model, image, ids):
    x = model.embed(ids)
    return x if image is None else torch.cat([image.double(), x])


# ------------------------------------------------------------------------------------ cases


def listed():
    seq = {"target": "llava7b", "layers": 4, "draft": "115m", "image": 576, "prompt": 64, "greedy": False}
    return [
        # the rule alone for one sequence: the smallest call there is
        {"name": "reject b1", "kind": "reject", "B": 1, "gamma": 5, "V": VOCAB, "sigma": 0.5, "greedy": False},
        # ... for a batch of sequences, with greedy decoding, closely matched draft
        {"name": "reject b32 greedy", "kind": "reject", "B": 32, "gamma": 5, "V": VOCAB, "sigma": 0.1, "greedy": True},
        # one block's gamma draft rows and gamma + 1 target rows through top-k / top-p
        {"name": "truncate 11 rows", "kind": "truncate", "rows": 11, "V": VOCAB, "top_k": 50, "top_p": 0.9},
        # a QKV-sized linear map on a verify block's rows
        {"name": "skinny bf16 qkv", "kind": "skinny", "M": 6, "N": 12288, "K": 4096, "dtype": "bf16", "noalloc": False},
        # a small fp32 map without allocation, as inside a latency-critical loop
        {"name": "skinny fp32 small", "kind": "skinny", "M": 4, "N": 688, "K": 256, "dtype": "fp32", "noalloc": True},
        # one image's 576 vision features into the target's space
        {"name": "adapter 576", "kind": "adapter", "m": 576, "d_in": 1024, "d_hid": 4096, "d_out": 4096},
        # time to the first token: 576 image rows + 64 prompt ids
        dict(seq, name="prefill 640", kind="prefill"),
        # the draft's five steps of a block
        dict(seq, name="draft g5", kind="draft", layers=1, gamma=5),
        # the verification step, sampling, part of the block accepted
        dict(seq, name="verify g5", kind="verify", gamma=5),
        # a small token tree, drafted and verified
        dict(seq, name="tree 2-1-1", kind="tree", layers=2, branching="2,1,1"),
        # 16 sequences with long caches, one block each
        dict(seq, name="batch 16x1600", kind="batch", B=16, gamma=5, prompt=1024),
        # the whole loop on the small fp32 models, prompt of 16 image rows and 16 ids
        {"name": "generate tiny", "kind": "generate", "target": "tiny", "draft": "tiny", "image": 16, "prompt": 16,
         "greedy": True, "gamma": 4, "new": 32},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["reject", "truncate", "skinny", "adapter", "prefill", "draft", "verify", "tree", "batch", "generate"])
    c = {"kind": kind}
    if kind == "reject":
        c.update(B=_log(rng, 1, 32), gamma=rng.randint(1, 7), V=_log(rng, 1000, VOCAB), sigma=rng.choice([0.1, 0.5, 1.0]),
                 greedy=rng.random() < 0.3)
    elif kind == "truncate":
        c.update(rows=_log(rng, 1, 96), V=_log(rng, 1000, VOCAB), top_k=rng.choice([0, 1, _log(rng, 2, 500)]),
                 top_p=rng.choice([1.0, 0.9, round(rng.uniform(0.3, 0.99), 3)]))
    elif kind == "skinny":
        noalloc = rng.random() < 0.4
        c.update(M=rng.randint(1, 8), N=_log(rng, 100, 900 if noalloc else 12288), K=8 * _log(rng, 16, 512),
                 dtype=rng.choice(["bf16", "bf16", "fp32"]), noalloc=noalloc)
    elif kind == "adapter":
        wide = rng.choice([1024, 4096, 8 * _log(rng, 32, 512)])
        c.update(m=_log(rng, 16, 576), d_in=rng.choice([1024, 8 * _log(rng, 16, 128)]), d_hid=wide, d_out=wide)
    elif kind == "generate":
        c.update(target="tiny", draft="tiny", image=rng.choice([0, 16]), prompt=_log(rng, 4, 48), greedy=rng.random() < 0.7,
                 gamma=rng.randint(0, 7), new=_log(rng, 8, 48))
    else:
        c.update(target="llava7b", layers=rng.randint(1, 3), draft=rng.choice(["115m", "115m", "table1"]),
                 image=rng.choice([0, 576, _log(rng, 16, 576)]), prompt=_log(rng, 16, 900), greedy=rng.random() < 0.4)
        if kind in ("draft", "verify"):
            c.update(gamma=rng.randint(1, 7))
            if not c["greedy"] and rng.random() < 0.3:
                c.update(top_k=50, top_p=0.9)
        elif kind == "tree":
            c.update(greedy=False, branching=rng.choice(["2,2", "3,1", "2,1,1", "7", "1,1,1", "1,2,1"]))
        elif kind == "batch":
            gamma = rng.randint(1, 7)
            c.update(gamma=gamma, B=_log(rng, 2, 16 if gamma < 7 else 15))
    return c


def _nodes(case):
    branching = [int(b) for b in case["branching"].split(",")]
    n, level = 0, 1
    for b in branching:
        level *= b
        n += level
    return branching, n


def _rows64(seed, rows, V):
    g = torch.Generator(DEV).manual_seed(seed)
    return torch.softmax(torch.randn(rows, V, generator=g, device=DEV) * 3.0, -1)


def _reject_inputs(case, seed):
    B, G, V = case["B"], case["gamma"], case["V"]
    g = torch.Generator(DEV).manual_seed(seed)
    t = torch.randn(B, G + 1, V, generator=g, device=DEV) * 3.0
    d = t[:, :G] + case["sigma"] * torch.randn(B, G, V, generator=g, device=DEV)
    p, q = torch.softmax(t, -1), torch.softmax(d, -1)
    ids = (q.argmax(-1) if case["greedy"] else
           torch.multinomial(q.view(B * G, V), 1, generator=g).view(B, G)).to(torch.int32).contiguous()
    u = torch.from_numpy(_uniforms(_rng(seed), B, G + 1)).to(DEV)
    return p, q, ids, u


def _skinny_inputs(case, seed):
    g = torch.Generator(DEV).manual_seed(seed)
    x = torch.randn(case["M"], case["K"], generator=g, device=DEV)
    w = torch.randn(case["N"], case["K"], generator=g, device=DEV) * 0.02
    return x, w.to(torch.bfloat16) if case["dtype"] == "bf16" else w


def _adapter_inputs(case, seed):
    g = torch.Generator(DEV).manual_seed(seed)
    h = torch.randn(case["m"], case["d_in"], generator=g, device=DEV)
    w1 = (torch.randn(case["d_hid"], case["d_in"], generator=g, device=DEV) * 0.02).to(torch.bfloat16)
    w2 = (torch.randn(case["d_out"], case["d_hid"], generator=g, device=DEV) * 0.02).to(torch.bfloat16)
    return h, w1, w2


def _verify_ids(case, seed, pending):
    """Draft ids of a verify call: some that the target agrees with, then others; q rows, uniforms."""
    G = case["gamma"]
    g = _rng(seed * 64 + 63)
    keep = int(g.integers(0, G + 1))
    ids = np.full(G, pending, dtype=np.int32)
    ids[keep:] = g.integers(0, VOCAB, size=G - keep)
    q = torch.softmax(torch.randn(G, VOCAB, generator=torch.Generator(DEV).manual_seed(seed), device=DEV), -1)
    return ids, q, _uniforms(g, G + 1)


def prepare(case, seed):
    kind, s = case["kind"], SimpleNamespace(case=case)
    if kind == "reject":
        s.p, s.q, s.ids, s.u = _reject_inputs(case, seed)
        s.n_acc, s.next = (torch.zeros(case["B"], dtype=torch.int32, device=DEV) for _ in range(2))
    elif kind == "truncate":
        s.probs = _rows64(seed, case["rows"], case["V"])
        s.out = torch.empty_like(s.probs)
    elif kind == "skinny":
        s.x, s.w = _skinny_inputs(case, seed)
        s.y = torch.empty(case["M"], case["N"], device=DEV)
    elif kind == "adapter":
        s.ctx = _context(dict(target="tiny", draft="tiny", greedy=True), 64, 1)
        s.h, s.w1, s.w2 = _adapter_inputs(case, seed)
        s.out = torch.empty(case["m"], case["d_out"], device=DEV)
    elif kind == "batch":
        G, B = case["gamma"], case["B"]
        lead = _context(case, case["image"] + case["prompt"] + 2 * (G + 1) + 1, G)
        s.seqs = [lead] + [lead.fork() for _ in range(B - 1)]
        s.at = []
        for b, c in enumerate(s.seqs):
            image, ids, u0, g = _sequence(case, seed, b)
            s.at.append((len(ids), int(ids[-1]), c.prefill(image, ids, u0)))
        s.batch = spd.SpdBatch(s.seqs)
        s.ud = torch.from_numpy(_uniforms(g, B, G)).to(DEV)
        s.uv = torch.from_numpy(_uniforms(g, B, G + 1)).to(DEV)
        s.logits = torch.empty(B * (G + 1), VOCAB, device=DEV)
    else:
        tc, _ = _models(case)
        _, nodes = _nodes(case) if kind == "tree" else (None, 0)
        G = {"tree": nodes, "prefill": 5}.get(kind, case.get("gamma"))
        s.ctx = _context(case, case["image"] + case["prompt"] + case.get("new", 0) + 2 * (G + 1) + 16, G)
        s.image, s.ids, s.u0, g = _sequence(case, seed)
        s.logits = torch.empty(1 if kind == "prefill" else G + 1, tc.vocab, device=DEV)
        if kind == "prefill":
            return s
        pending = s.ctx.prefill(s.image, s.ids, s.u0)
        s.at = (len(s.ids), int(s.ids[-1]), pending)
        if kind == "draft":
            s.u = _uniforms(g, G)
            s.probs = torch.zeros(G, tc.vocab, device=DEV)
            s.logits = s.logits[: min(6, G)]     # the library keeps the last six rows
        elif kind == "verify":
            s.draft_ids, s.q, s.u = _verify_ids(case, seed, pending)
        elif kind == "tree":
            s.branching, _ = _nodes(case)
            s.ud, s.uv = _uniforms(g, nodes), _uniforms(g, nodes + 1)
        else:
            s.u = _uniforms(g, case["new"], 2 * G + 1)
    return s


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "reject":
        spd.reject_sample(s.p, s.q, s.ids, s.u, case["gamma"], case["greedy"], s.n_acc, s.next)
        return {"n_accepted": s.n_acc, "next": s.next}
    if kind == "truncate":
        spd.truncate_probs(s.probs, s.out, case["top_k"], case["top_p"])
        return s.out
    if kind == "skinny":
        gemm = spd.skinny_gemm_noalloc if case["noalloc"] else spd.skinny_gemm
        gemm(s.x, s.w, s.y, 1 if case["dtype"] == "bf16" else 0)
        return s.y
    if kind == "adapter":
        return s.ctx.image_adapter(s.h, s.w1, s.w2, s.out)
    if kind == "prefill":
        first = s.ctx.prefill(s.image, s.ids, s.u0)
        return {"logits": _logits(s.ctx, s.logits), "token": first}
    if kind == "draft":   # the draft starts from the committed text each time
        ids = s.ctx.draft(case["gamma"], s.u, None if case["greedy"] else s.probs)
        s.ctx._check(spd.lib().spd_get_draft_logits(s.ctx._ctx, _ptr(s.logits), int(s.logits.shape[0])))
        return {"logits": s.logits, "ids": ids} if case["greedy"] else {"logits": s.logits, "probs": s.probs, "ids": ids}
    if kind == "batch":
        for c, at in zip(s.seqs, s.at):   # every pass decodes the block behind the prompt
            c.rollback(*at)
        ids = s.batch.draft(case["gamma"], s.ud)
        n_acc, nxt = s.batch.verify(case["gamma"], s.uv)
        s.batch._check(spd.lib().spd_batch_get_logits(s.batch._bt, _ptr(s.logits), int(s.logits.shape[0])))
        return {"logits": s.logits, "draft_ids": ids, "n_accepted": n_acc, "next": nxt}
    s.ctx.rollback(*s.at)
    if kind == "verify":
        n_acc, nxt = s.ctx.verify(case["gamma"], s.u, s.draft_ids, s.q)
        return {"logits": _logits(s.ctx, s.logits), "n_accepted": n_acc, "next": nxt}
    if kind == "tree":
        parent, ids = s.ctx.draft_tree(s.branching, s.ud)
        path, nxt = s.ctx.verify_tree(parent, s.uv)
        return {"logits": _logits(s.ctx, s.logits), "node_ids": ids, "path": np.asarray(path, dtype=np.int64), "next": nxt}
    out, _ = s.ctx.generate(case["new"], case["gamma"], s.u)
    return {"ids": out, "logits": _logits(s.ctx, s.logits)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "reject":
        return None
    if kind == "truncate":
        return torch.stack([_truncate64(r, case["top_k"], case["top_p"]) for r in _rows64(seed, case["rows"], case["V"])])
    if kind == "skinny":
        x, w = _skinny_inputs(case, seed)
        return x.double() @ w.double().T
    if kind == "adapter":
        h, w1, w2 = (t.double() for t in _adapter_inputs(case, seed))
        a = h @ w1.T
        return (0.5 * a * (1 + torch.erf(a / math.sqrt(2.0)))) @ w2.T
    if kind == "generate" and not case["greedy"]:
        return None     # which tokens the last block holds depends on every draw before it
    tc, dc = _models(case)
    target = _Model64(tc, WEIGHT_SEED)
    if kind == "generate":
        # the loop ends with the block that reaches `new` tokens: its rows are those behind the last commit
        return None if case["gamma"] else _generate64(case, seed, target)
    draft = _Model64(dc, WEIGHT_SEED + 1) if kind in ("draft", "batch", "tree") else None

    def drafted(text, uniforms):
        ids, rows = [], []
        for u in uniforms:
            row = draft.logits(draft.embed(text + ids), 1)[0]
            rows.append(row)
            ids.append(_token64(case, row, float(u)))
        return ids, torch.stack(rows)

    if kind == "batch":
        G, rows = case["gamma"], []
        seqs = [_sequence(case, seed, b) for b in range(case["B"])]
        ud = _uniforms(seqs[-1][3], case["B"], G)
        for (image, ids, u0, _), u in zip(seqs, ud):
            x = _prompt64(target, image, ids)
            text = [int(t) for t in ids] + [_token64(case, target.logits(x, 1)[0], u0)]
            block, _ = drafted(text, u)
            rows.append(target.logits(_prompt64(target, image, text + block), G + 1))
        return {"logits": torch.cat(rows), "draft_ids": None, "n_accepted": None, "next": None}
    image, ids, u0, g = _sequence(case, seed)
    first = target.logits(_prompt64(target, image, ids), 1)
    if kind == "prefill":
        return {"logits": first, "token": None}
    pending = _token64(case, first[0], u0)
    text = [int(t) for t in ids] + [pending]
    if kind == "draft":
        _, rows = drafted(text, _uniforms(g, case["gamma"]))
        if case["greedy"]:
            return {"logits": rows[:6], "ids": None}
        return {"logits": rows[:6], "probs": _probs64(case, rows), "ids": None}
    if kind == "verify":
        block, _, _ = _verify_ids(case, seed, pending)
        rows = target.logits(_prompt64(target, image, text + [int(t) for t in block]), case["gamma"] + 1)
        return {"logits": rows, "n_accepted": None, "next": None}
    # tree: node i's row is the last row of the chain of its ancestors
    branching, n = _nodes(case)
    ud, paths, chains, level = _uniforms(g, n), [[]], [[]], [0]
    for b in branching:
        grown = []
        for node in level:
            row = draft.logits(draft.embed(text + chains[node]), 1)[0]
            for _ in range(b):
                grown.append(len(chains))
                chains.append(chains[node] + [_token64(case, row, float(ud[len(chains) - 1]))])
        level = grown
    rows = torch.cat([target.logits(_prompt64(target, image, text + c), 1) for c in chains])
    return {"logits": rows, "node_ids": None, "path": None, "next": None}


def _generate64(case, seed, target):
    image, ids, _, _ = _sequence(case, seed)
    text, row = [int(t) for t in ids], None
    for _ in range(case["new"]):
        row = target.logits(_prompt64(target, image, text), 1)
        text.append(int(row[0].argmax()))
    return {"ids": None, "logits": row}


def _layer_params(c):
    return c.n_layers * (4 * c.d_model ** 2 + 3 * c.d_model * c.d_ffn)


def _pass_work(c, rows, cached, head_rows, weights=True):
    """One forward of `rows` new rows of a model behind `cached` cached rows: weights read once, cache rows
    read and written once, logits written."""
    b = 2 if c.dtype == "bf16" else 4
    par, head = _layer_params(c), c.vocab * c.d_model * (1 if head_rows else 0)
    kv = 2 * c.n_layers * c.d_model * b
    attended = rows * cached + rows * (rows + 1) / 2
    return ((par + head) * b * weights + kv * (cached + rows) + 4 * c.vocab * head_rows,
            2.0 * par * rows + 2.0 * head * head_rows + 4.0 * c.n_layers * c.d_model * attended)


def work(case):
    kind = case["kind"]
    if kind == "reject":   # the rows the rule has to look at: one pair, or with greedy decoding one row per test
        n = case["gamma"] + 1 if case["greedy"] else 2
        return {"bytes": 4.0 * case["B"] * case["V"] * n, "flops": 2.0 * case["B"] * case["V"] * n}
    if kind == "truncate":
        return {"bytes": 8.0 * case["rows"] * case["V"], "flops": 4.0 * case["rows"] * case["V"]}
    if kind == "skinny":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": N * K * (2.0 if case["dtype"] == "bf16" else 4.0) + 4.0 * M * (N + K), "flops": 2.0 * M * N * K}
    if kind == "adapter":
        m, i, h, o = case["m"], case["d_in"], case["d_hid"], case["d_out"]
        return {"bytes": 2.0 * (i * h + h * o) + 4.0 * m * (i + o), "flops": 2.0 * m * (i * h + h * o)}
    tc, dc = _models(case)
    rows, text = case["image"] + case["prompt"], case["prompt"]
    if kind == "prefill":
        t, d = _pass_work(tc, rows, 0, 1), _pass_work(dc, text, 0, 0)
        return {"bytes": t[0] + d[0] + 4.0 * rows * tc.d_model, "flops": t[1] + d[1]}
    G = case.get("gamma", 0)
    if kind == "draft":
        b, f = _pass_work(dc, 1, text + 1, 1)
        return {"bytes": G * b, "flops": G * f}
    if kind == "verify":
        b, f = _pass_work(tc, G + 1, rows, G + 1)
        return {"bytes": b, "flops": f}
    if kind == "tree":
        branching, n = _nodes(case)
        b, f = _pass_work(tc, n + 1, rows, n + 1)
        level = 1
        for k in branching:
            x, y = _pass_work(dc, level, text + 1, level)
            b, f, level = b + x, f + y, level * k
        return {"bytes": b, "flops": f}
    if kind == "batch":
        b = f = 0.0
        for i in range(case["B"]):   # the weights once for all sequences
            x, y = _pass_work(tc, G + 1, rows, G + 1, i == 0)
            v, w = _pass_work(dc, 1, text + 1, 1, i == 0)
            b, f = b + x + G * v, f + y + G * w
        return {"bytes": b, "flops": f}
    blocks = -(-(case["new"] - 1) // (G + 1))   # every block accepted
    t, d = _pass_work(tc, G + 1, rows, G + 1), _pass_work(dc, 1, text, 1)
    return {"bytes": blocks * (t[0] + G * d[0]), "flops": blocks * (t[1] + G * d[1])}


def tolerance(case):
    kind = case["kind"]
    if kind in ("reject", "truncate"):
        return "exact"      # integer masses: no order of summation shows
    if kind == "skinny":
        return {"rel": 2e-5 if case["dtype"] == "bf16" else 1e-6}
    if kind == "adapter":
        return {"rel": 5e-5}    # two maps of activations split into two bf16 parts: 1.2e-5 off 64 bits
    if kind == "generate":
        return {"rel": 1e-5}
    return {"rel": 1e-3}        # K and V are cached in bf16: 1e-4 to 2.5e-4 off 64 bits
