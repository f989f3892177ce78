"""The work a user of this library has it do, as cases that can be timed and checked.

Four kinds of case, each one call (or one request) through the public entry points:

* ``attention`` -- the stand-alone tree-attention operator (``esp_tree_attention``) on caller-owned buffers;
* ``step``      -- one synchronous decode-and-verify step of a handle whose sequences are prefilled (the cache grows
                   by the emitted tokens from pass to pass, as it does in a serving loop);
* ``prefill``   -- ``esp_prefill`` of one prompt (time to first token);
* ``request``   -- ``Handle.generate``: prefill and synchronous steps until the requested tokens have been emitted.

Model cases return the emitted tokens and, through ``esp_debug_capture``, the logits of the rows whose content does not
depend on which drafts the previous step proposed: the root row and, where only the root carries a probe chain, the
probe rows.

Weights.  Embeddings N(0, 1), matrices N(0, 0.02^2) with the residual branches' output matrices scaled by
1/sqrt(2 * layers) (the usual initialisation of deep decoders), and an LM head whose row pi(v) points along the
embedding of v, with pi a permutation of one long cycle, or of short cycles.  Trained models have peaked next-token
distributions; these weights have one too, so that the emitted stream does not hang on the last bit of a logit.
With one long cycle no draft is ever right (1 token per step); with cycles of 4 tokens the static tree's first depth
always holds the right token (2 tokens per step).  The tiny fp32 model keeps its plain N(0, 0.02^2) tied weights.
"""
import math

import numpy as np
import torch

import paper_2603_17942_b200 as P
import synth

R = P.ESP_MAX_ROWS
SMALL = synth.TINY.replace(name="bf16-small", dtype="bf16", tied=False, n_layers=3, d_model=512, n_q_heads=4,
                           n_kv_heads=2, head_dim=128, d_ffn=688, vocab=5000)
SHAPES = {"tiny-fp32": synth.TINY, "bf16-small": SMALL, "llama3-8b": synth.LLAMA3_8B, "qwen3-8b": synth.QWEN3_8B}
STEP_ROOM = 2048       # positions a step case's sequences can grow by before they are prefilled again


def listed():
    return [
        # the operator on one sequence: the smallest call, latency counts (32/8 heads of 128, 64-node tree + 4 probes)
        dict(name="attention-b1-4k", kind="attention", dtype="bf16", batch=1, kv=4096, heads=32, kv_heads=8, head_dim=128, nodes=64, probes=4),
        # the same operator on a serving batch
        dict(name="attention-b16-4k", kind="attention", dtype="bf16", batch=16, kv=4096, heads=32, kv_heads=8, head_dim=128, nodes=64, probes=4),
        # full-precision heads of the tiny model, a ragged cache length
        dict(name="attention-fp32", kind="attention", dtype="fp32", batch=3, kv=777, heads=4, kv_heads=2, head_dim=64, nodes=32, probes=3),
        # the tiny fp32 decoder's whole request: 64-token prompt, 64 tokens, trees of at most 32 nodes
        dict(name="tiny-fp32-request", kind="request", model="tiny-fp32", layers=2, prompt=64, new=64, batch=1, k=3, topk=4, nodes=32, tree="root", cycle=0, temperature=0.0),
        # a small bf16 decoder with sample matching: launches and latency count
        dict(name="small-bf16-sampled", kind="request", model="bf16-small", layers=3, prompt=150, new=32, batch=1, k=3, topk=5, nodes=16, tree="root", cycle=0, temperature=1.0),
        # the headline: one step of the 8B decoder behind a 1024-token prompt, 64-node tree + 4 probes
        dict(name="llama3-8b-step", kind="step", model="llama3-8b", layers=32, prompt=1024, batch=1, k=4, topk=10, nodes=64, tree="root", cycle=0, temperature=0.0),
        # a whole request of the other 8B decoder (per-head norms, larger vocabulary), 2048-token prompt
        dict(name="qwen3-8b-request", kind="request", model="qwen3-8b", layers=36, prompt=2048, new=16, batch=1, k=4, topk=8, nodes=48, tree="root", cycle=0, temperature=0.0),
        # time to first token of a long prompt (8 of the 32 layers)
        dict(name="llama-prefill-8k", kind="prefill", model="llama3-8b", layers=8, prompt=8192, batch=1, k=4, topk=10, nodes=64, tree="root", cycle=0, temperature=0.0),
        # several sequences per step (8 of the 32 layers)
        dict(name="llama-step-b4-4k", kind="step", model="llama3-8b", layers=8, prompt=4096, batch=4, k=4, topk=10, nodes=64, tree="root", cycle=0, temperature=0.0),
        # the largest serving batch at a long context (4 of the 32 layers)
        dict(name="llama-step-b8-16k", kind="step", model="llama3-8b", layers=4, prompt=16384, batch=8, k=4, topk=10, nodes=64, tree="root", cycle=0, temperature=0.0),
        # probes behind every node: the paper's largest block, 120 rows
        dict(name="llama-step-bc120", kind="step", model="llama3-8b", layers=8, prompt=1024, batch=1, k=3, topk=10, nodes=30, tree="every", cycle=0, temperature=0.0),
        # a short request with the static tree [7, 2] and accepted drafts (2 tokens per step)
        dict(name="llama-static-accepting", kind="request", model="llama3-8b", layers=8, prompt=333, new=24, batch=1, k=2, topk=7, nodes=10, tree="static", cycle=4, temperature=0.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["attention", "attention", "step", "step", "prefill", "request"])
    if kind == "attention":
        if rng.random() < 0.25:
            return dict(kind=kind, dtype="fp32", batch=rng.randint(1, 4), kv=_log(rng, 16, 2048), heads=4, kv_heads=2,
                        head_dim=64, nodes=rng.randint(1, 40), probes=rng.randint(0, 4))
        batch = _log(rng, 1, 16)
        return dict(kind=kind, dtype="bf16", batch=batch, kv=_log(rng, 64, 65536 // batch), heads=32, kv_heads=8,
                    head_dim=128, nodes=rng.randint(1, 120), probes=rng.randint(0, 8))
    model = rng.choice(["bf16-small", "llama3-8b", "llama3-8b", "qwen3-8b"] + (["tiny-fp32"] if kind != "prefill" else []))
    big = model.endswith("8b")
    tree = rng.choice(["root", "root", "every", "static"])
    if tree == "root":
        k, topk, nodes = rng.randint(3, 4), rng.randint(4, 10), rng.randint(8, 64)
    elif tree == "every":
        k, topk, nodes = 3, rng.randint(4, 10), rng.randint(8, 30)
    else:
        k, topk, nodes = 2, 7, 10
    c = dict(kind=kind, model=model, layers=rng.randint(1, 6) if big else SHAPES[model].n_layers, batch=1, k=k, topk=topk,
             nodes=nodes, tree=tree, cycle=4 if tree == "static" and model != "tiny-fp32" and kind == "request" else 0,
             temperature=rng.choice([0.0, 0.0, 1.0]) if model != "tiny-fp32" else 0.0)
    if kind == "step":
        c["batch"] = rng.randint(1, 8) if model != "tiny-fp32" else rng.randint(1, 2)
        c["prompt"] = _log(rng, 32, min(16384, 32768 // c["batch"])) if big else _log(rng, 16, 1024)
    elif kind == "prefill":
        c["prompt"] = _log(rng, 32, 8192) if big else _log(rng, 16, 2048)
    else:
        c["prompt"], c["new"] = _log(rng, 32, 2048) if big else _log(rng, 8, 512), rng.randint(4, 48)
    return c


# ---------------------------------------------------------------- inputs
def _shape(case):
    return SHAPES[case["model"]].replace(n_layers=case["layers"])


def _spec(case, seed):
    base = dict(n_probes=case["k"], temperature=case["temperature"], seed=seed)
    if case["tree"] == "static":
        return P.spec_cfg(topk=case["topk"], max_nodes=case["nodes"], n_anchor=0, static_widths=(7, 2), **base)
    if case["tree"] == "every":
        return P.spec_cfg(topk=case["topk"], max_nodes=case["nodes"], expand_width=1, n_anchor=0, **base)
    return P.spec_cfg(topk=case["topk"], max_nodes=case["nodes"], expand_width=0, n_anchor=1, **base)


def _successor(case, vocab, seed):
    """pi as an int64 array: one cycle over the vocabulary, or cycles of case["cycle"] tokens."""
    order = np.random.default_rng(seed + 5).permutation(vocab)
    c = case["cycle"] or vocab
    nxt = np.empty(vocab, np.int64)
    for s in ([0] if c == vocab else range(c)):
        if c == vocab:
            nxt[order] = np.roll(order, -1)
        else:
            whole = vocab // c * c
            block = order[:whole].reshape(-1, c)
            nxt[block[:, s]] = block[:, (s + 1) % c]
            nxt[order[whole:]] = order[whole:]
    return nxt


def _weights(case, shape, seed):
    w = synth.make_weights(shape, seed, device="cuda")
    if shape.tied:
        return w, None
    nxt = _successor(case, shape.vocab, seed)
    w["embed"] = (w["embed"].float() * 50).to(torch.bfloat16)
    head = torch.empty_like(w["lm_head"])
    head[torch.from_numpy(nxt).cuda()] = (w["embed"].float() * (80.0 / shape.d_model)).to(torch.bfloat16)
    w["lm_head"] = head
    for name in ("wo", "w_down"):
        for t in w[name]:
            t.copy_(t.float() / math.sqrt(2 * shape.n_layers))
    return w, nxt


def _prompts(case, vocab, seed):
    return [synth.make_prompt(vocab, case["prompt"], seed * 64 + i) for i in range(case["batch"])]


def _attention_inputs(case, seed):
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    B, Hq, Hkv, h, L = case["batch"], case["heads"], case["kv_heads"], case["head_dim"], case["kv"]
    M = case["nodes"] + case["probes"]
    cap = L + R
    q, kc, vc, kb, vb = synth.random_qkv((B, R, Hq, h), (B, Hkv, cap, h), (B, Hkv, M, h), seed, "cuda", dt)
    kc[:, :, L:L + M] = kb
    vc[:, :, L:L + M] = vb
    vis = np.zeros((B, R, R), bool)
    depth = np.zeros((B, R), np.int32)
    for s in range(B):
        parents = synth.random_tree_parents(case["nodes"], 5, seed * 64 + s)
        for i, p in enumerate(parents):
            vis[s, i, i] = True
            if p >= 0:
                vis[s, i] |= vis[s, p]
                depth[s, i] = depth[s, p] + 1
        for j in range(case["probes"]):                      # the root's probe chain
            r = case["nodes"] + j
            vis[s, r, 0] = True
            vis[s, r, case["nodes"]:r + 1] = True
            depth[s, r] = j + 1
        for r in range(M, R):
            vis[s, r, r] = True
    anc = np.packbits(vis, axis=-1, bitorder="little").view(np.int64).reshape(B, R, 2)
    return q, kc, vc, torch.from_numpy(anc).cuda(), torch.from_numpy(depth).cuda(), vis, depth, M


class _Model:
    pass


def prepare(case, seed):
    if case["kind"] == "attention":
        q, kc, vc, anc, depth, _, _, M = _attention_inputs(case, seed)
        cap = case["kv"] + R
        nb = P.esp_tree_attention_scratch_bytes(case["batch"], case["heads"], case["head_dim"], cap)
        return dict(case=case, q=q, kc=kc, vc=vc, anc=anc, depth=depth, M=M, out=torch.zeros_like(q), nb=nb,
                    scratch=torch.empty(nb, dtype=torch.uint8, device="cuda"))
    shape = _shape(case)
    s = _Model()
    s.case, s.shape = case, shape
    w, _ = _weights(case, shape, seed)
    s.prompts = _prompts(case, shape.vocab, seed)
    s.logits = torch.zeros(case["batch"] * R, shape.vocab, dtype=torch.float32, device="cuda")
    s.stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    new = case.get("new", 0)
    room = STEP_ROOM if case["kind"] == "step" else (new + case["k"] + 1)
    s.handle = P.Handle(shape, _spec(case, seed), w, case["prompt"] + room, case["batch"], s.stream)
    P.esp_debug_capture(s.handle.h, s.logits)
    if case["kind"] == "step":
        _refill(s)
    return s


def _refill(s):
    for i, p in enumerate(s.prompts):
        s.handle.prefill(p, i)
    s.handle.step()
    s.left = STEP_ROOM // (s.case["k"] + 1) - 2


def _rows(s, kind):
    """The captured rows that do not depend on earlier drafts, and the last forward's layout."""
    v = s.logits.view(s.case["batch"], R, -1)
    k = s.case["k"]
    if kind == "prefill":
        last = (s.case["prompt"] - 1) % P.ESP_PREFILL_CHUNK
        return v[:, last:last + 1 + k]
    if s.case["tree"] == "root":
        n = s.case["nodes"]
        return v[:, 0], v[:, n:n + k]
    return v[:, 0]


def run(s):
    if isinstance(s, dict):
        c = s["case"]
        P.esp_tree_attention(1 if c["dtype"] == "bf16" else 0, c["batch"], s["M"], c["kv"], c["kv"] + R, c["heads"], c["kv_heads"],
                             c["head_dim"], 16, s["q"], s["kc"], s["vc"], s["anc"], s["depth"], s["out"], s["scratch"],
                             s["nb"], torch.cuda.current_stream().cuda_stream)
        return s["out"][:, :s["M"]]
    if s.case["kind"] == "prefill":
        first = s.handle.prefill(s.prompts[0])
        return {"token": first, "logits": _rows(s, "prefill")}
    if s.case["kind"] == "request":
        tokens = s.handle.generate(s.prompts[0], s.case["new"])
        return {"tokens": np.array(tokens, np.int64), "logits": _rows(s, "step")}
    if s.left <= 0:
        _refill(s)
    s.handle.step()
    s.left -= 1
    h = s.handle
    tokens = np.where(np.arange(h.tokens_out.shape[1])[None] < h.n_out[:, None], h.tokens_out, -1)
    return {"tokens": tokens.astype(np.int64), "logits": _rows(s, "step")}


# ---------------------------------------------------------------- what a pass cannot do without
def _rows_of(case):
    if case["tree"] == "root":
        return case["nodes"] + case["k"]
    return (case["k"] + 1) * case["nodes"]


def _model_work(case, rows, kv, tokens_streamed):
    """One forward of `rows` rows per sequence over a cache of `kv` positions, all sequences."""
    s = _shape(case)
    es = 4 if s.dtype == "fp32" else 2
    b = case["batch"]
    d, dq, dkv = s.d_model, s.n_q_heads * s.head_dim, s.n_kv_heads * s.head_dim
    layer = d * dq + 2 * d * dkv + dq * d + 3 * d * s.d_ffn
    flops = 2.0 * b * rows * layer * s.n_layers + 4.0 * b * rows * kv * dq * s.n_layers
    byts = (layer * s.n_layers + s.vocab * d) * es + 2.0 * b * kv * dkv * es * s.n_layers
    return byts, flops + 2.0 * b * tokens_streamed * s.vocab * d


def work(case):
    if case["kind"] == "attention":
        es = 2 if case["dtype"] == "bf16" else 4
        M, h = case["nodes"] + case["probes"], case["head_dim"]
        byts = case["batch"] * es * h * (2 * case["kv_heads"] * (case["kv"] + M) + 2 * M * case["heads"])
        return {"bytes": byts, "flops": 4.0 * case["batch"] * M * case["heads"] * (case["kv"] + 6) * h}
    rows = _rows_of(case)
    if case["kind"] == "step":
        b, f = _model_work(case, rows, case["prompt"] + 1, rows)
        return {"bytes": b, "flops": f}
    b, f = _model_work(case, case["prompt"], case["prompt"] / 2, 1 + case["k"])
    if case["kind"] == "request":
        steps = (case["new"] - 1) // (2 if case["cycle"] else 1)
        b2, f2 = _model_work(case, rows, case["prompt"] + case["new"] / 2, rows)
        b, f = b + steps * b2, f + steps * f2
    return {"bytes": b, "flops": f}


def tolerance(case):
    """fp32: sums in another order (6e-7 from 64 bits).  bf16: the operator's result, a number rounded to bf16 from
    bf16 probabilities, is 2.3e-3 from 64 bits; the logits are 2e-3 to 1e-2 away (the longer the prefill the more: the
    cache, the queries and the attention weights are bf16), and two correct implementations differ by as much."""
    if case.get("dtype") == "fp32" or case.get("model") == "tiny-fp32":
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 1e-2 if case["kind"] == "attention" else 2e-2, "max": 2e-1}


# ---------------------------------------------------------------- the same in 64 bits
def _rope(x, pos, base):
    half = x.shape[-1] // 2
    inv = base ** (-torch.arange(half, dtype=torch.float64, device=x.device) / half)
    a = pos.double()[:, None] * inv[None]
    c, s = a.cos()[:, None], a.sin()[:, None]
    lo, hi = x[..., :half], x[..., half:]
    return torch.cat([lo * c - hi * s, hi * c + lo * s], -1)


def _norm(x, g, eps):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * g.double()


def _logits64(shape, w, tokens, extra, first_row):
    """Logits of rows first_row.. of the causal sequence embed[tokens] + extra vectors."""
    x = torch.cat([w["embed"][torch.as_tensor(tokens, device="cuda")].double(), extra])
    T, h, g = x.shape[0], shape.head_dim, shape.n_q_heads // shape.n_kv_heads
    pos = torch.arange(T, device="cuda")
    for l in range(shape.n_layers):
        y = _norm(x, w["norm_attn"][l], shape.rms_eps)
        q = (y @ w["wq"][l].double().T).view(T, -1, h)
        k = (y @ w["wk"][l].double().T).view(T, -1, h)
        v = (y @ w["wv"][l].double().T).view(T, -1, h)
        if shape.qk_norm:
            q, k = _norm(q, w["q_norm"][l], shape.rms_eps), _norm(k, w["k_norm"][l], shape.rms_eps)
        q, k = _rope(q, pos, shape.rope_base), _rope(k, pos, shape.rope_base)
        o = torch.empty_like(q)
        for r0 in range(0, T, 1024):
            r1 = min(T, r0 + 1024)
            block = pos[r0:r1, None] < pos[None, :r1]
            for j in range(shape.n_kv_heads):
                sc = torch.einsum("rgd,cd->grc", q[r0:r1, j * g:(j + 1) * g], k[:r1, j]) / math.sqrt(h)
                sc.masked_fill_(block[None], -math.inf)
                o[r0:r1, j * g:(j + 1) * g] = torch.einsum("grc,cd->rgd", torch.softmax(sc, -1), v[:r1, j])
        x = x + o.reshape(T, -1) @ w["wo"][l].double().T
        y = _norm(x, w["norm_ffn"][l], shape.rms_eps)
        x = x + (torch.nn.functional.silu(y @ w["w_gate"][l].double().T) * (y @ w["w_up"][l].double().T)) @ w["w_down"][l].double().T
    return _norm(x[first_row:], w["final_norm"], shape.rms_eps) @ w["lm_head"].double().T


def _mask(shape, w, prompt, emitted, k, lam=0.1):
    m = w["embed"][torch.as_tensor(prompt, device="cuda", dtype=torch.long)].double().mean(0)
    for y in emitted:
        m = (1 - np.float64(np.float32(lam))) * m + np.float64(np.float32(lam)) * w["embed"][int(y)].double()
    return m[None].expand(k, -1)


def _attention64(case, seed):
    q, kc, vc, _, _, vis, depth, M = _attention_inputs(case, seed)
    B, L, h, g = case["batch"], case["kv"], case["head_dim"], case["heads"] // case["kv_heads"]
    out = torch.empty(B, M, case["heads"], h, dtype=torch.float64, device="cuda")
    for b in range(B):
        see = torch.ones(M, L + M, dtype=torch.bool, device="cuda")
        see[:, L:] = torch.from_numpy(vis[b, :M, :M]).cuda()
        for j in range(case["kv_heads"]):
            sc = torch.einsum("rgd,cd->grc", q[b, :M, j * g:(j + 1) * g].double(), kc[b, j, :L + M].double()) / math.sqrt(h)
            sc.masked_fill_(~see[None], -math.inf)
            out[b, :, j * g:(j + 1) * g] = torch.einsum("grc,cd->rgd", torch.softmax(sc, -1), vc[b, j, :L + M].double())
    return out


def exact(case, seed):
    if case["kind"] == "attention":
        return _attention64(case, seed)
    shape = _shape(case)
    n = case["prompt"] + (case.get("new", 2))
    layer = shape.n_params_streamed() - shape.vocab * shape.d_model
    flops = case["batch"] * (2.0 * n * layer + 2.0 * n * n * shape.n_q_heads * shape.head_dim * shape.n_layers)
    if flops > 1.5e14:
        return None
    w, nxt = _weights(case, shape, seed)
    k = case["k"]
    steps = {"prefill": 0, "step": 2, "request": case.get("new", 0) - 1}[case["kind"]]
    tokens, root, probes = [], [], []
    for prompt in _prompts(case, shape.vocab, seed):
        seq = [int(t) for t in prompt]
        none = torch.zeros(0, shape.d_model, dtype=torch.float64, device="cuda")
        for _ in range(steps):                                # the tokens before the last forward
            seq.append(int(nxt[seq[-1]]) if nxt is not None else int(_logits64(shape, w, seq, none, len(seq) - 1)[0].argmax()))
        # a prefill draws its probe rows from the prompt's mean, a step from the mask after all emitted tokens
        got = _logits64(shape, w, seq, _mask(shape, w, prompt, seq[len(prompt):], k), len(seq) - 1)
        last = int(nxt[seq[-1]]) if nxt is not None else int(got[0].argmax())
        tokens.append(seq[len(prompt):] + [last])
        root.append(got[:1])
        probes.append(got[1:])
    if case["kind"] == "prefill":
        return {"token": tokens[0][0], "logits": torch.stack([torch.cat([root[0], probes[0]])])}
    rows = None if case["cycle"] else torch.cat(root)       # with accepted drafts the last root depends on the steps' sizes
    if case["tree"] == "root":
        rows = [rows, torch.stack(probes)]
    if case["kind"] == "request":
        return {"tokens": np.array(tokens[0], np.int64), "logits": rows}
    last = np.full((case["batch"], P.ESP_MAX_PROBES + 1), -1, np.int64)
    last[:, 0] = [t[-1] for t in tokens]
    return {"tokens": last, "logits": rows}
