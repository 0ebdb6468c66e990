"""What the speed of this framework is measured on: its linears and attention layers through
the stateless entry points, and whole calls (prefill, draft-and-verify steps, plain
autoregressive steps) through the context API.

listed() are the measured cases, draw() gives more of the same ranges; prepare() builds what a
program holds before the call, run() is one pass, exact() the same numbers in 64 bits.
Shapes are those of the repository's configurations: the 4096-wide 32-layer model (32 heads of
128, FFN 11008, vocabulary 32000) in bf16, the 5120-wide one for its layers, the 512-wide
two-layer bf16 one and the 256-wide two-layer fp32 one.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2402_15758_gb300 as pkg

STD = 0.02  # standard deviation of every weight

MODELS = {
    "fp32_256": dict(n_layers=2, d_model=256, n_heads=4, head_dim=64, ffn_dim=688, vocab=1024, dtype="fp32",
                     topk=[4, 2, 1, 1]),
    "bf16_512": dict(n_layers=2, d_model=512, n_heads=4, head_dim=128, ffn_dim=1408, vocab=2048, dtype="bf16",
                     topk=[5, 5, 5, 5]),
    "bf16_4096": dict(n_layers=32, d_model=4096, n_heads=32, head_dim=128, ffn_dim=11008, vocab=32000,
                      dtype="bf16", topk=[5, 5, 5, 5]),
}
for _m in MODELS.values():
    _m.update(rms_eps=1e-6, rope_theta=10000.0, n_draft_heads=4, kv_block=16)


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------
def _linear(name, rows, n, k, epi, split=True, dtype="bf16", out="fp32"):
    return dict(name=name, kind="linear", rows=rows, n=n, k=k, epi=epi, split=split, dtype=dtype, out=out)


def _attention(name, batch, heads, head_dim, queries, n_local, q_local0, ctx_min, ctx_max, splits, split=True,
               dtype="bf16"):
    return dict(name=name, kind="attention", batch=batch, heads=heads, head_dim=head_dim, queries=queries,
                n_local=n_local, q_local0=q_local0, ctx_min=ctx_min, ctx_max=ctx_max, splits=splits, split=split,
                dtype=dtype)


def _model(name, kind, model, batch, prompt_min, prompt_max, nodes, steps):
    return dict(name=name, kind=kind, model=model, batch=batch, prompt_min=prompt_min, prompt_max=prompt_max,
                nodes=nodes, steps=steps)


def listed():
    return [
        # the smallest call: one projection of a few rows at odd sizes, bf16 result
        _linear("linear_small_ragged", 5, 1000, 520, 1, split=False, out="bf16"),
        # a residual decoding head of the draft: one row against the vocabulary
        _linear("linear_head_1row", 1, 32000, 8192, 0),
        # SwiGLU's gate and up projections for a 64-node tree, added to the output
        _linear("linear_gate_up_64row", 64, 22016, 4096, 2),
        # the down projection for 8 sequences of 32 nodes
        _linear("linear_down_256row", 256, 4096, 11008, 2),
        # an attention layer (attention and output projection) of the draft: one query
        _attention("attention_draft_1query", 1, 32, 128, 1, 4, 3, 512, 512, 4),
        # ... of the verification of a 64-node tree at an ordinary context
        _attention("attention_tree_64", 1, 32, 128, 64, 64, 0, 1000, 1000, 4),
        # ... of a ragged batch of 32-node trees
        _attention("attention_batch8_ragged", 8, 32, 128, 32, 32, 0, 256, 4096, 2),
        # ... at a long context
        _attention("attention_tree_16k", 1, 32, 128, 64, 64, 0, 16384, 16384, 4),
        # a whole small request in fp32: prompt and eight steps, all latency and launches
        _model("request_fp32_256", "request", "fp32_256", 1, 64, 64, 16, 8),
        # a prompt of the 4096-wide model, whole
        _model("prefill_4096", "prefill", "bf16_4096", 1, 600, 600, 64, 0),
        # decoding at batch 1: draft-and-verify steps of a 64-node tree
        _model("steps_4096", "steps", "bf16_4096", 1, 512, 512, 64, 4),
        # batched serving: 8 ragged sequences, 32-node trees
        _model("steps_4096_batch8", "steps", "bf16_4096", 8, 256, 4096, 32, 2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["linear", "attention", "request", "prefill", "steps", "ar"], [8, 7, 2, 1, 1, 1])[0]
    if kind == "linear":
        dtype = rng.choices(["bf16", "fp32"], [5, 1])[0]
        if dtype == "fp32":  # the layers of the fp32 model
            return dict(kind=kind, rows=_log_int(rng, 1, 64), n=4 * _log_int(rng, 64, 512), k=_log_int(rng, 128, 1024),
                        epi=rng.choice([0, 1, 2]), split=False, dtype=dtype, out="fp32")
        epi = rng.choice([0, 1, 2])
        return dict(kind=kind, rows=_log_int(rng, 1, 512), n=_log_int(rng, 500, 32000),
                    k=8 * _log_int(rng, 64, 1536), epi=epi, split=rng.random() < 0.75, dtype=dtype,
                    out="fp32" if epi == 2 or rng.random() < 0.5 else "bf16")
    if kind == "attention":
        heads, head_dim, dtype = rng.choice([(32, 128, "bf16"), (32, 128, "bf16"), (40, 128, "bf16"), (4, 64, "fp32")])
        batch = _log_int(rng, 1, 8)
        tree = rng.random() < 0.7
        nodes = rng.randint(2, 64 if batch == 1 else 32)
        ctx = _log_int(rng, 64, 16384 // batch if dtype == "bf16" else 512)
        return dict(kind=kind, batch=batch, heads=heads, head_dim=head_dim, queries=nodes if tree else 1,
                    n_local=nodes if tree else 4, q_local0=0 if tree else 3, ctx_min=max(1, ctx // 3), ctx_max=ctx,
                    splits=rng.randint(1, 8), split=dtype == "bf16" and rng.random() < 0.8, dtype=dtype)
    if kind == "request":
        model = rng.choice(["fp32_256", "bf16_512"])
        batch = rng.randint(1, 4)
        prompt = _log_int(rng, 8, 400)
        return dict(kind=kind, model=model, batch=batch, prompt_min=max(1, prompt // 2), prompt_max=prompt,
                    nodes=rng.randint(4, 16 if model == "fp32_256" else 64), steps=rng.randint(1, 8))
    if kind == "prefill":
        batch = rng.randint(1, 3)
        prompt = _log_int(rng, 24, 1000 // batch)
        return dict(kind=kind, model="bf16_4096", batch=batch, prompt_min=max(1, prompt // 2), prompt_max=prompt,
                    nodes=64, steps=0)
    batch = rng.randint(1, 4)
    prompt = _log_int(rng, 64, 2000)
    return dict(kind=kind, model="bf16_4096", batch=batch, prompt_min=max(1, prompt // 2), prompt_max=prompt,
                nodes=rng.randint(16, 64 if batch == 1 else 32), steps=rng.randint(1, 4))


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(g, shape, std, dtype):
    return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=g)


def _between(lo, hi, count, seed):
    r = np.random.default_rng(seed)
    return [int(v) for v in r.integers(lo, hi + 1, count)]


def _two_terms(x32):
    hi = x32.to(torch.bfloat16)
    return hi, (x32 - hi.float()).to(torch.bfloat16)


def _linear_inputs(c, seed):
    g = _generator(seed)
    dt = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    x32 = _normal(g, (c["rows"], c["k"]), 1.0, torch.float32)
    s = dict(x=x32.to(dt), x_lo=None, w=_normal(g, (c["n"], c["k"]), STD, dt))
    if c["split"]:
        s["x"], s["x_lo"] = _two_terms(x32)
    out = torch.float32 if c["out"] == "fp32" else torch.bfloat16
    s["y"] = _normal(g, (c["rows"], c["n"]), 1.0, out)  # the residual stream that epilogue 2 adds to
    return s


def _tree_masks(n, q_local0, r):
    """Ancestor-or-self masks: a random tree, or the causal chain of the draft's rows."""
    parent = [-1] + [int(r.integers(0, j)) for j in range(1, n)] if q_local0 == 0 else list(range(-1, n - 1))
    masks = []
    for i in range(n):
        masks.append((masks[parent[i]] if parent[i] >= 0 else 0) | (1 << i))
    return masks


def _attention_inputs(c, seed):
    g, r = _generator(seed), np.random.default_rng(seed)
    B, H, hd = c["batch"], c["heads"], c["head_dim"]
    dt = torch.float32 if c["dtype"] == "fp32" else torch.bfloat16
    ctx = _between(c["ctx_min"], c["ctx_max"], B, seed)
    pages = (max(ctx) + c["n_local"] + 15) // 16
    blocks = B * pages
    kv = _normal(g, (blocks, H, 2, 16, hd), 1.0, torch.float32)
    if c["split"]:
        hi, lo = _two_terms(kv)
        pool = torch.stack([hi[:, :, 0], lo[:, :, 0], hi[:, :, 1], lo[:, :, 1]], 2).contiguous()
        del hi, lo
    else:
        pool = kv.to(dt)
    masks = _tree_masks(c["n_local"], c["q_local0"], r)
    rows, d = B * c["queries"], H * hd
    return dict(kv=kv, pool=pool, ctx=ctx, masks=masks, table=torch.from_numpy(r.permutation(blocks).astype(np.int32)).reshape(B, pages).cuda(),
                n_ctx=torch.tensor(ctx, dtype=torch.int32, device="cuda"),
                anc=torch.from_numpy(np.array(masks, dtype=np.uint64).view(np.int64)).cuda(),
                q=_normal(g, (rows, d), 1.0, torch.float32), wo=_normal(g, (d, d), STD, dt),
                x=_normal(g, (rows, d), 1.0, torch.float32),
                out=torch.empty(rows, d, dtype=dt, device="cuda"),
                out_lo=torch.empty(rows, d, dtype=dt, device="cuda") if c["split"] else None)


def _config(c):
    return dict(MODELS[c["model"]], tree_nodes=c["nodes"], batch=c["batch"])


def _weights(cfg, seed):
    g = _generator(seed)
    d, f, v = cfg["d_model"], cfg["ffn_dim"], cfg["vocab"]
    dt = torch.float32 if cfg["dtype"] == "fp32" else torch.bfloat16
    # a trained model's token scores are uneven: rows of the heads differ in size, so the best
    # token leads by more than rounding can move it
    size = torch.exp(0.5 * _normal(g, (v, 1), 1.0, torch.float32)).to(dt)
    w = {"embed": _normal(g, (v, d), STD, dt), "lm_head": _normal(g, (v, d), STD, dt) * size,
         "tri_w1": _normal(g, (d, 3 * d), STD, dt), "tri_w2": _normal(g, (d, d), STD, dt)}
    for b in [f"layers.{i}" for i in range(cfg["n_layers"])] + ["draft"]:
        for name, shape in (("wqkv", (3 * d, d)), ("wo", (d, d)), ("w_gate", (f, d)), ("w_up", (f, d)),
                            ("w_down", (d, f))):
            w[f"{b}.{name}"] = _normal(g, shape, STD, dt)
        for name in ("attn_norm", "ffn_norm"):
            w[f"{b}.{name}"] = 1.0 + 0.1 * _normal(g, (d,), 1.0, dt)
    w["final_norm"] = 1.0 + 0.1 * _normal(g, (d,), 1.0, dt)
    for k in range(cfg["n_draft_heads"]):
        w[f"heads.{k}"] = _normal(g, (v, 2 * d), STD, dt) * size
    return w


def _prompts(c, cfg, seed):
    r = np.random.default_rng(seed)
    return [r.integers(0, cfg["vocab"], n).tolist() for n in _between(c["prompt_min"], c["prompt_max"], c["batch"], seed)]


ROOM = 2000  # tokens a sequence can grow by while its state is stepped again and again


def prepare(case, seed):
    c = case
    if c["kind"] == "linear":
        return dict(_linear_inputs(c, seed), case=c)
    if c["kind"] == "attention":
        s = dict(_attention_inputs(c, seed), case=c)
        del s["kv"]
        return s
    cfg = _config(c)
    prompts = _prompts(c, cfg, seed)
    room = 128 + 8 * 5 if c["kind"] in ("request", "prefill") else ROOM
    seq = (max(len(p) for p in prompts) + room + 15) // 16 * 16
    model = pkg.Chimera(cfg, _weights(cfg, seed), max_batch=c["batch"], max_seq_len=seq)
    if c["kind"] in ("steps", "ar"):
        model.prefill(prompts)
    return dict(case=c, model=model, prompts=prompts)


# ---------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------
def _padded(rows, width):
    out = np.full((len(rows), width), -1, np.int64)
    for b, r in enumerate(rows):
        out[b, :len(r)] = r
    return out


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "linear":
        pkg.op_linear(s["x"], s["w"], s["y"], epi=c["epi"], out_f32=c["out"] == "fp32", X_lo=s["x_lo"])
        return s["y"]
    if c["kind"] == "attention":  # the attention and the output projection, added to the residual stream
        pkg.op_attention(s["q"], s["pool"], s["table"], s["n_ctx"], s["anc"], s["out"], nq=c["queries"],
                         q_local0=c["q_local0"], n_local=c["n_local"], q_rows=c["queries"], n_heads=c["heads"],
                         head_dim=c["head_dim"], splits=c["splits"], out_lo=s["out_lo"])
        pkg.op_linear(s["out"], s["wo"], s["x"], epi=2, out_f32=True, X_lo=s["out_lo"])
        return s["x"]
    m = s["model"]
    if c["kind"] == "prefill":  # the scores of each prompt's next token
        m.prefill(s["prompts"])
        return m.read("prefill_logits")
    if c["kind"] == "ar":  # tokens and the scores of the last one
        tokens = m.ar_generate(c["steps"])
        return dict(tokens=_padded(tokens, c["steps"]), logits=m.read("prefill_logits"))
    if c["kind"] == "request":
        m.prefill(s["prompts"])
    # the emitted tokens and the last step's scores.  Those of the draft's heads, which rest on the
    # hidden state that the step before verified, come always; those of the tree's nodes where a
    # model is small: over 32 layers rounding (5e-5) can swap two nodes whose drafted tokens are
    # nearly tied (in one step out of a hundred), and their rows with them
    tokens = m.generate(c["steps"])
    r = dict(tokens=_padded(tokens, 5 * c["steps"]), draft_logits=m.read("draft_logits"))
    if c["kind"] == "request":
        r["verify_logits"] = m.read("verify_logits")
    return r


# ---------------------------------------------------------------------------------------
# what a pass cannot do without, and how exactly it is defined
# ---------------------------------------------------------------------------------------
def _esize(c):
    return 4 if c["dtype"] == "fp32" else 2


def work(case):
    c = case
    if c["kind"] == "linear":
        e, terms = _esize(c), 2 if c["split"] else 1
        y = c["rows"] * c["n"] * (4 if c["out"] == "fp32" else 2)
        return {"bytes": c["n"] * c["k"] * e + c["rows"] * c["k"] * e * terms + y * (2 if c["epi"] == 2 else 1),
                "flops": 2.0 * c["rows"] * c["n"] * c["k"] * terms}
    if c["kind"] == "attention":
        e, terms = _esize(c), 2 if c["split"] else 1
        d, rows = c["heads"] * c["head_dim"], c["batch"] * c["queries"]
        keys = c["batch"] * ((c["ctx_min"] + c["ctx_max"]) / 2 + c["n_local"])
        return {"bytes": keys * d * 2 * e * terms + rows * d * 4 + d * d * e + rows * d * 8,
                "flops": 4.0 * c["queries"] * keys * d * (3 if c["split"] else 1) + 2.0 * rows * d * d * terms}
    cfg = MODELS[c["model"]]
    e = 4 if cfg["dtype"] == "fp32" else 2
    d, f, v, L, K = cfg["d_model"], cfg["ffn_dim"], cfg["vocab"], cfg["n_layers"], cfg["n_draft_heads"]
    B, n = c["batch"], (c["prompt_min"] + c["prompt_max"]) / 2
    terms = 1 if cfg["dtype"] == "fp32" else 2
    layer = 4 * d * d + 3 * d * f
    kv = 2 * d * e * terms  # a position's keys and values in one layer

    def pass_(rows, ctx_keys, logit_rows):  # a base forward of `rows` rows over `ctx_keys` cached positions
        return np.array([L * layer * e + v * d * e + rows * d * e + L * (ctx_keys + rows) * kv,
                         2.0 * terms * (rows * L * layer + logit_rows * v * d)])

    prompt = pass_(B * n, 0, B) + [0, 4.0 * L * d * B * n * n / 2 * (1.5 * terms)]
    draft = np.array([K * (4 * d * d + layer) * e + K * v * 2 * d * e + K * B * n * kv,
                      2.0 * terms * B * K * (4 * d * d + layer + 2 * v * d)])
    step = draft + pass_(B * c["nodes"], B * n, B * c["nodes"])
    total = {"prefill": prompt, "ar": c["steps"] * pass_(B, B * n, B), "steps": c["steps"] * step,
             "request": prompt + c["steps"] * step}[c["kind"]]
    return {"bytes": float(total[0]), "flops": float(total[1])}


def tolerance(case):
    """About four times the error against exact() at the start, or the change of a whole model's
    scores between two runs (fp32 sums in another order), whichever is larger."""
    c = case
    if c["kind"] == "linear":
        if c["out"] == "bf16":  # one rounding to bf16: 1.7e-3
            return {"rel": 6e-3, "max": 2e-2}
        # fp32 sums of up to 12288 products in the tensor cores: 1.6e-5 at 8192
        return {"rel": 6e-5, "max": 1e-3} if c["dtype"] == "bf16" else {"rel": 4e-6, "max": 4e-5}
    if c["kind"] == "attention":
        if c["split"] or c["dtype"] == "fp32":  # 7e-7, the projection's share of a residual stream
            return {"rel": 5e-6, "max": 1e-4}
        return {"rel": 2e-3, "max": 2e-2}  # the attention's output is rounded once to bf16: 3e-4
    if MODELS[c["model"]]["dtype"] == "fp32":  # 3e-7
        return {"rel": 2e-6, "max": 4e-5, "differ": 0.0}
    return {"rel": 5e-4, "max": 5e-3, "differ": 0.0}  # 1.2e-4 after 32 layers


# ---------------------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------------------
def _exact_linear(c, seed):
    s = _linear_inputs(c, seed)
    x = s["x"].double() + (s["x_lo"].double() if c["split"] else 0.0)
    y = torch.cat([x @ w.double().T for w in s["w"].split(4096)], 1)
    if c["epi"] == 1:
        y = y * torch.sigmoid(y)
    return s["y"].double() + y if c["epi"] == 2 else y


def _exact_attention(c, seed):
    s = _attention_inputs(c, seed)
    B, H, hd, nq = c["batch"], c["heads"], c["head_dim"], c["queries"]
    kv = s["kv"] if c["split"] or c["dtype"] == "fp32" else s["pool"].float()
    q = s["q"].double().view(B, nq, H, hd)
    outs = []
    for b in range(B):
        n, slots = s["ctx"][b], s["ctx"][b] + c["n_local"]
        own = kv[s["table"][b].long()]  # [pages][H][2][16][hd]
        o = torch.empty(nq, H, hd, dtype=torch.float64, device="cuda")
        seen = torch.zeros(nq, slots, dtype=torch.bool, device="cuda")
        seen[:, :n] = True
        for i in range(nq):
            for j in range(c["n_local"]):
                if s["masks"][c["q_local0"] + i] >> j & 1:
                    seen[i, n + j] = True
        for h in range(H):
            k = own[:, h, 0].reshape(-1, hd)[:slots].double()
            v = own[:, h, 1].reshape(-1, hd)[:slots].double()
            a = (q[b, :, h] @ k.T / math.sqrt(hd)).masked_fill(~seen, -math.inf)
            o[:, h] = torch.softmax(a, -1) @ v
        outs.append(o.reshape(nq, H * hd))
    return s["x"].double() + torch.cat(outs) @ s["wo"].double().T


def _best_ranks(topk, nodes):
    """The static tree: the rank tuples with the largest product of the heads' accuracies."""
    acc = [(66, 78, 83, 87, 90), (49, 55, 60, 68, 75), (38, 44, 49, 55, 62), (33, 38, 43, 46, 54)]
    gain = [[a[0]] + [a[i] - a[i - 1] for i in range(1, 5)] for a in acc]
    tuples = [((), 100 ** 4)]
    for h, lim in enumerate(topk):
        tuples += [(t + (r,), p // 100 * gain[h][r]) for t, p in tuples if len(t) == h for r in range(min(lim, 5))]
    best = sorted(tuples[1:], key=lambda x: (-x[1], len(x[0]), x[0]))[:nodes - 1]
    return [()] + sorted((t for t, _ in best), key=lambda t: (len(t), t))


class _Exact:
    """The model in 64 bits, one sequence, every forward from scratch."""

    def __init__(self, cfg, w):
        self.cfg, self.w = cfg, w
        self.inv = cfg["rope_theta"] ** (-torch.arange(0, cfg["head_dim"], 2, dtype=torch.float64, device="cuda")
                                         / cfg["head_dim"])

    def norm(self, x, g):
        return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + self.cfg["rms_eps"]) * self.w[g].double()

    def lin(self, x, name):
        return torch.cat([x @ w.double().T for w in self.w[name].split(8192)], -1)

    def rope(self, x, pos):
        a = pos.double()[:, None] * self.inv
        c, s = a.cos()[:, None], a.sin()[:, None]
        u, v = x.chunk(2, -1)
        return torch.cat([u * c - v * s, v * c + u * s], -1)

    def block(self, x, name, pos, seen, keys=None):
        """One block over rows x; `seen` over their own keys, after `keys` (normed inputs and positions of others)."""
        cfg = self.cfg
        n, d, H, hd = x.shape[0], cfg["d_model"], cfg["n_heads"], cfg["head_dim"]
        q, k, v = self.lin(self.norm(x, name + ".attn_norm"), name + ".wqkv").view(n, 3, H, hd).unbind(1)
        q, k = self.rope(q, pos), self.rope(k, pos)
        if keys is not None:
            kv = self.norm(keys[0], name + ".attn_norm") @ self.w[name + ".wqkv"][d:].double().T
            k0, v0 = kv.view(-1, 2, H, hd).unbind(1)
            k, v = torch.cat([self.rope(k0, keys[1]), k]), torch.cat([v0, v])
        a = torch.einsum("qhd,khd->hqk", q, k) / math.sqrt(hd)
        a = torch.softmax(a.masked_fill(~seen, -math.inf), -1)
        x = x + self.lin(torch.einsum("hqk,khd->qhd", a, v).reshape(n, d), name + ".wo")
        h = self.norm(x, name + ".ffn_norm")
        gate = self.lin(h, name + ".w_gate")
        return x + self.lin(gate * torch.sigmoid(gate) * self.lin(h, name + ".w_up"), name + ".w_down")

    def base(self, tokens, pos, seen):
        x = self.w["embed"][torch.tensor(tokens, device="cuda")].double()
        for i in range(self.cfg["n_layers"]):
            x = self.block(x, f"layers.{i}", pos, seen)
        return self.norm(x, "final_norm")

    def causal(self, tokens):
        n = len(tokens)
        return self.base(tokens, torch.arange(n, device="cuda"),
                         torch.ones(n, n, dtype=torch.bool, device="cuda").tril())

    def draft(self, tokens, hidden):
        """The heads' scores after `tokens` (the last one the root), hidden of all but the root."""
        cfg, n, x, logits = self.cfg, hidden.shape[0], list(tokens), []
        tri = torch.empty(0, cfg["d_model"], dtype=torch.float64, device="cuda")
        for k in range(cfg["n_draft_heads"]):
            e = [self.w["embed"][x[i]].double() if i >= 0 else torch.zeros(cfg["d_model"], device="cuda").double()
                 for i in range(n + k - 2, n + k + 1)]
            u = self.lin(torch.cat(e)[None], "tri_w1")
            tri = torch.cat([tri, self.lin(u * torch.sigmoid(u), "tri_w2")])
            seen = torch.ones(k + 1, n + k + 1, dtype=torch.bool, device="cuda").tril(n)
            full = self.block(tri, "draft", torch.arange(n, n + k + 1, device="cuda"), seen,
                              (hidden, torch.arange(n, device="cuda")))
            logits.append(self.lin(torch.cat([hidden[-1], full[-1]])[None], f"heads.{k}")[0])
            x.append(int(logits[-1].argmax()))
        return torch.stack(logits)


def _exact_model(c, seed):
    cfg = _config(c)
    weights = cfg["n_layers"] * (4 * cfg["d_model"] ** 2 + 3 * cfg["d_model"] * cfg["ffn_dim"])
    passes = 2 if c["kind"] == "prefill" else (2 + c["steps"])
    if 2.0 * weights * c["batch"] * passes / 2 * (c["prompt_max"] + c["nodes"]) > 1.2e13:
        return None
    w = _weights(cfg, seed)
    m = _Exact(cfg, w)
    ranks = _best_ranks(cfg["topk"], c["nodes"])
    first, tokens, draft, verify = [], [], [], []
    for x in _prompts(c, cfg, seed):
        x = list(x)
        first.append(m.lin(m.causal(x)[-1:], "lm_head")[0])
        if c["kind"] == "prefill":
            continue
        out = []
        x.append(int(first[-1].argmax()))
        for _ in range(c["steps"]):  # x: the committed tokens and the root
            n = len(x) - 1
            if c["kind"] == "ar":
                first[-1] = m.lin(m.causal(x)[-1:], "lm_head")[0]
                out.append(x[-1])
                x.append(int(first[-1].argmax()))
                continue
            # the tree's tokens need the draft's scores, and those only the hidden rows before the root
            d = m.draft(x, m.causal(x[:-1]))
            top = d.topk(5, -1).indices.tolist()
            toks = [x[-1]] + [top[len(t) - 1][t[-1]] for t in ranks[1:]]
            pos = torch.tensor(list(range(n)) + [n + len(t) for t in ranks], device="cuda")
            seen = torch.zeros(n + len(ranks), n + len(ranks), dtype=torch.bool, device="cuda")
            seen[:n, :n] = torch.ones(n, n, dtype=torch.bool, device="cuda").tril()
            seen[n:, :n] = True
            for i, t in enumerate(ranks):
                for j, u in enumerate(ranks):
                    seen[n + i, n + j] = t[:len(u)] == u
            v = m.lin(m.base(x[:-1] + toks, pos, seen)[n:], "lm_head")
            want, at = v.argmax(-1).tolist(), 0
            path = [0]
            while True:
                kids = [j for j, t in enumerate(ranks) if len(t) == len(ranks[at]) + 1 and t[:-1] == ranks[at]]
                hit = [j for j in kids if toks[j] == want[at]]
                if not hit:
                    break
                at = hit[0]
                path.append(at)
            out += [toks[j] for j in path]
            x = x[:-1] + [toks[j] for j in path] + [want[at]]
        tokens.append(out)
        if c["kind"] != "ar":
            draft.append(d)
            verify.append(v)
    if c["kind"] == "prefill":
        return torch.stack(first)
    if c["kind"] == "ar":
        return dict(tokens=None, logits=torch.stack(first))
    r = dict(tokens=None, draft_logits=torch.stack(draft, 1))
    if c["kind"] == "request":
        r["verify_logits"] = torch.stack(verify)
    return r


def exact(case, seed):
    """`run`'s outputs in 64 bits; None for models and prompts that would take too long."""
    if case["kind"] == "linear":
        return _exact_linear(case, seed)
    if case["kind"] == "attention":
        return _exact_attention(case, seed)
    return _exact_model(case, seed)
