"""Performance cases of the draft-and-verify decode loop, through the package's public entry points.

A case is a dict of plain values; `listed()` holds the fixed ones, `draw(rng)` makes one more of the same ranges,
`prepare` builds what a program has in hand before the call, `run` makes one pass, `work` says what a pass cannot do
without, `tolerance` how far another correct implementation may be off, and `exact` is the same pass in 64 bits
with plain torch.

Kinds of cases (`op`):
  request  a prompt (or a ragged batch of them) is processed and `steps` draft-and-verify steps follow
  decode   the prompts are in the cache already; a pass is `steps` further steps
  prefill  prompt processing alone
  linear   the single projection y = x W^T
  labels   the training-label matrix of a batch of samples

The decoder's weights are synthetic but peaked, as a trained model's are: the embedding dominates the residual
stream and row t of lm_head is a sum of the embeddings of the tokens 1, 2, ... places before t in a fixed cyclic
order, with falling weights. So the model's next token stands out, the extra heads rank the tokens after it, and a
step accepts two or three tokens. That keeps every accepted token far from a tie: another order of the sums does not
change the stream, and hidden states and logits of two implementations can be compared.
"""
import math
import random

import numpy as np
import torch

from paper_2503_14153_b200 import FLAG_KEEP_LOGITS, SpecDecoder, build_tree, spec_build_labels, spec_op_linear
from paper_2503_14153_b200.binding import DBG_H_LAST, DBG_LOGITS, DBG_NEXT_ROOT
from synthetic.configs import ModelConfig

DEVICE = "cuda:0"
STRIDE = 977                                   # tokens follow one another in steps of STRIDE (mod vocab)
LEVELS = [1.0] + [0.5 * 0.88 ** i for i in range(9)]   # how strongly lm_head points to the 1st, 2nd, ... next token
PAD, IGNORE, FRAG = 0, -100, 7
TYP_EPS, TYP_DELTA = 0.09, 0.3

# widths of the repository's configurations and tests: (d_model, heads, kv heads, head_dim, ffn)
WIDE = dict(dtype="bf16", d=4096, heads=32, kv=32, hd=128, ffn=11008, vocab=32016)
MEDIUM = dict(dtype="bf16", d=1024, heads=16, kv=4, hd=64, ffn=2752, vocab=32016)
NARROW = dict(dtype="bf16", d=512, heads=4, kv=4, hd=128, ffn=1344, vocab=3000)
TINY = dict(dtype="fp32", d=256, heads=4, kv=4, hd=64, ffn=688, vocab=32016)
DRAFT4 = dict(topk="10,4,2,2")
DRAFT3 = dict(topk="4,2,2")


def _loop(name, op, width, layers, lo, hi, batch=1, nodes=64, steps=1, topk="10,4,2,2", p=-1.0, temperature=0.0, logits=False):
    c = dict(op=op, **width, layers=layers, topk=topk, nodes=nodes, batch=batch, prompt_lo=lo, prompt_hi=hi, steps=steps,
             p=p, temperature=temperature, logits=logits)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # a small float32 model answering a short prompt: launches and latency are all there is
        _loop("tiny_fp32_request", "request", TINY, 2, 32, 32, nodes=16, steps=24, topk="4,2,2"),
        # one user of the full 7B shape: a 256-token prompt and the start of its answer, 64-node tree
        _loop("7b_request", "request", WIDE, 32, 256, 256, steps=24),
        # candidates supplied by another draft model (override table), small tree, logits read for scoring
        _loop("7b_controlled_draft_logits", "decode", WIDE, 2, 512, 512, nodes=16, steps=16, p=0.6, logits=True),
        # decoding far into a long context (a quarter of the 7B depth)
        _loop("7b_long_context", "decode", WIDE, 8, 8192, 8192, steps=4),
        # batched serving: 16 ragged sequences, 1024 rows to verify a step (a quarter of the depth)
        _loop("7b_batch16", "decode", WIDE, 8, 128, 2048, batch=16),
        # a long prompt to its first token
        _loop("7b_prefill_2048", "prefill", WIDE, 8, 2048, 2048),
        # ragged prompts admitted together
        _loop("7b_prefill_batch8", "prefill", WIDE, 4, 128, 1024, batch=8),
        # grouped-query heads of 64, three sequences, a tree that is no multiple of a tile
        _loop("gqa_batch3_request", "request", MEDIUM, 6, 37, 411, batch=3, nodes=23, steps=16),
        # sampled decoding with typical acceptance, the second decoding mode of the method
        _loop("7b_sampled_request", "request", WIDE, 4, 256, 256, steps=8, temperature=0.8),
        # one projection at the rows of a 64-node tree, and at those of a batch
        dict(name="linear_bf16_m64", op="linear", dtype="bf16", m=64, n=11008, k=4096),
        dict(name="linear_bf16_m1008", op="linear", dtype="bf16", m=1008, n=11008, k=4096),
        # labels of a training batch, ten heads
        dict(name="labels_256x2048", op="labels", seqs=256, length=2048, heads=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choices(["wide", "medium", "narrow", "tiny", "prefill", "linear", "labels"], [3, 2, 1, 1, 2, 2, 1])[0]
    if kind == "labels":
        return dict(op="labels", seqs=_log(rng, 1, 256), length=_log(rng, 16, 4000), heads=rng.randint(0, 16))
    if kind == "linear":
        if rng.random() < 0.25:
            return dict(op="linear", dtype="fp32", m=_log(rng, 1, 100), n=_log(rng, 100, 3000), k=8 * _log(rng, 8, 128))
        return dict(op="linear", dtype="bf16", m=16 * _log(rng, 1, 96), n=_log(rng, 128, 12000), k=64 * _log(rng, 2, 172))
    if kind == "prefill":
        width, layers = rng.choice([(WIDE, rng.randint(1, 4)), (MEDIUM, rng.randint(1, 8))])
        batch = rng.choice([1, 1, 1, rng.randint(2, 8)])
        hi = _log(rng, 16, 4096) if batch == 1 else _log(rng, 32, 1024)
        return _loop("", "prefill", width, layers, hi if batch == 1 else max(8, hi // 8), hi, batch=batch)
    width, layers = {"wide": (WIDE, rng.randint(1, 4)), "medium": (MEDIUM, rng.randint(1, 8)),
                     "narrow": (NARROW, rng.randint(1, 6)), "tiny": (TINY, rng.randint(1, 3))}[kind]
    if kind == "wide" and rng.random() < 0.3:
        width = dict(width, kv=8)
    if kind == "tiny":
        return _loop("", "request", width, layers, *([_log(rng, 4, 200)] * 2), nodes=_log(rng, 1, 26), steps=_log(rng, 4, 24), topk="4,2,2")
    batch = rng.choice([1, 1, 1, rng.randint(2, 4), rng.randint(2, 16)])
    nodes = rng.choice([1, 16, 32, 64, 128, rng.randint(2, 128)])
    hi = _log(rng, 16, 6000) if batch == 1 else _log(rng, 32, 1024)
    lo = hi if batch == 1 else max(8, hi // 8)
    long = hi > 1024 or batch > 4
    return _loop("", "decode" if long else "request", width, layers, lo, hi, batch=batch, nodes=nodes,
                 steps=rng.randint(1, 3) if long else rng.randint(2, 10), topk=rng.choice(["10,4,2,2", "10,4,2,2", "4,3,2,2,2,1,1,1,1,1"]) if nodes <= 48 else "10,4,2,2")


# ---------------------------------------------------------------- inputs
def _caps(case):
    return [int(v) for v in case["topk"].split(",")]


def _config(case):
    return ModelConfig(name="case", n_layers=case["layers"], d_model=case["d"], n_heads=case["heads"], n_kv_heads=case["kv"],
                       head_dim=case["hd"], d_ffn=case["ffn"], vocab=case["vocab"], rms_eps=1e-5, rope_base=1e6 if case["dtype"] == "bf16" else 1e4,
                       dtype=case["dtype"], n_medusa=len(_caps(case)), topk=tuple(_caps(case)), tree_nodes=case["nodes"],
                       prompt_len=case["prompt_hi"], new_tokens=0, seed=0, batch=case["batch"], norm_gain="random")


def _weights(case, seed):
    """Device tensors in the layout the decoder takes, drawn on the GPU from the seed."""
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    d, F, V, L = case["d"], case["ffn"], case["vocab"], case["layers"]
    hd, hq, hkv = case["hd"], case["heads"], case["kv"]
    g = torch.Generator(device=DEVICE).manual_seed(seed)

    def normal(rows, cols, std):
        return torch.randn((rows, cols), generator=g, device=DEVICE, dtype=dt).mul_(std)

    def gain():
        return 1.0 + 0.1 * torch.randn(d, generator=g, device=DEVICE)

    w = {"embed": normal(V, d, 1.0)}
    head = torch.zeros((V, d), device=DEVICE)
    for i, a in enumerate(LEVELS):
        head.add_(torch.roll(w["embed"], STRIDE * (i + 1), 0), alpha=0.02 * a)
    w["lm_head"] = head.to(dt)
    del head
    w["final_norm"] = gain()
    out_std = 0.02 / math.sqrt(2 * L) * math.sqrt(4096 / d)
    in_std = 0.02 * math.sqrt(4096 / d)
    for l in range(L):
        p = f"layers.{l}."
        w[p + "wqkv"] = normal((hq + 2 * hkv) * hd, d, in_std)
        w[p + "wo"] = normal(d, hq * hd, out_std)
        w[p + "w_gate"] = normal(F, d, in_std)
        w[p + "w_up"] = normal(F, d, in_std)
        w[p + "w_down"] = normal(d, F, out_std)
        w[p + "attn_norm"] = gain()
        w[p + "ffn_norm"] = gain()
    for k in range(len(_caps(case))):
        w[f"medusa.{k}.w"] = normal(d, d, in_std / 2)
        w[f"medusa.{k}.b"] = normal(1, d, 0.02)[0].contiguous()
    return w


def _prompts(case, seed):
    """Uniform random token ids; ragged lengths spread evenly over [prompt_lo, prompt_hi] in a random order."""
    rng = np.random.default_rng(np.random.SeedSequence([seed, 1]))
    lo, hi, n = case["prompt_lo"], case["prompt_hi"], case["batch"]
    lens = [hi] if n == 1 else [lo + round((hi - lo) * i / (n - 1)) for i in range(n)]
    rng.shuffle(lens)
    return [rng.integers(0, case["vocab"], size=int(m)).astype(np.int32) for m in lens]


def _tables(case, seed, prompts):
    """Override tables of the controlled draft (one a step): with probability p a head's first candidate is the token the
    model will say there, everything else is random. None where the heads' own candidates are used."""
    if case["p"] < 0:
        return None
    rng = np.random.default_rng(np.random.SeedSequence([seed, 2]))
    K, kmax, V = len(_caps(case)), _kmax(case), case["vocab"]
    return rng.integers(0, V, size=(64, case["batch"], K, kmax)).astype(np.int32), rng.random((64, case["batch"], K)) < case["p"]


def _tree(case):
    return build_tree(_caps(case), case["nodes"])


def _kmax(case):
    return int(max(_tree(case)["rank"])) + 1


def _override(case, tables, k, roots):
    t = tables[0][k % 64].copy()
    ahead = (roots[:, None].astype(np.int64) + STRIDE * (1 + np.arange(t.shape[1]))[None, :]) % case["vocab"]
    t[:, :, 0] = np.where(tables[1][k % 64], ahead, t[:, :, 0])
    return t


ROOM = 2048     # tokens a cache of a `decode` case can still take when it is made


def prepare(case, seed):
    if case["op"] == "labels":
        g = torch.Generator(device=DEVICE).manual_seed(seed)
        t = torch.randint(8, 32016, (case["seqs"], case["length"]), generator=g, device=DEVICE, dtype=torch.int32)
        t[torch.rand(t.shape, generator=g, device=DEVICE) < 0.15] = FRAG
        return dict(case=case, tokens=t)
    if case["op"] == "linear":
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        g = torch.Generator(device=DEVICE).manual_seed(seed)
        return dict(case=case, x=torch.randn((case["m"], case["k"]), generator=g, device=DEVICE, dtype=dt),
                    w=torch.randn((case["n"], case["k"]), generator=g, device=DEVICE, dtype=dt).mul_(0.02))
    cfg, prompts = _config(case), _prompts(case, seed)
    K = len(_caps(case))
    room = ROOM if case["op"] == "decode" else (K + 1) * (case["steps"] + 1)
    dec = SpecDecoder(cfg, _weights(case, seed), _tree(case), max_seq=case["prompt_hi"] + room, max_batch=case["batch"],
                      flags=FLAG_KEEP_LOGITS if case["logits"] else 0, accept_mode=1 if case["temperature"] > 0 else 0,
                      typ_eps=TYP_EPS, typ_delta=TYP_DELTA, temperature=case["temperature"] or 1.0,
                      sampling=case["temperature"] > 0, seed=seed)
    s = dict(case=case, dec=dec, prompts=prompts, tables=_tables(case, seed, prompts), k=0, used=0, room=room)
    if case["op"] == "decode":
        _admit(s)
    return s


def _admit(s):
    s["dec"].prefill(s["prompts"])
    s["used"] = 0
    if s["tables"] is not None:
        s["roots"] = s["dec"].debug(DBG_NEXT_ROOT)


def run(state):
    case = state["case"]
    if case["op"] == "labels":
        return spec_build_labels(state["tokens"], case["heads"], FRAG, PAD, IGNORE)
    if case["op"] == "linear":
        return spec_op_linear(state["x"], state["w"])
    dec, K = state["dec"], len(_caps(case))
    if case["op"] == "prefill":
        dec.prefill(state["prompts"])
        return dict(next=dec.debug(DBG_NEXT_ROOT), hidden=dec.debug(DBG_H_LAST))
    if case["op"] == "request":
        dec.prefill(state["prompts"])
    elif state["used"] + (K + 1) * (case["steps"] + 1) > state["room"]:
        _admit(state)                      # the sequence is full: the next one starts
    tokens, counts = [], []
    for _ in range(case["steps"]):
        ov = None
        if state["tables"] is not None:
            ov = _override(case, state["tables"], state["k"], state["roots"])
            state["k"] += 1
        t, n = dec.step(ov)
        if state["tables"] is not None:    # the model's next token, one place after the last it emitted
            last = t[np.arange(len(n)), n - 1]
            state["roots"] = ((last.astype(np.int64) + STRIDE) % case["vocab"]).astype(np.int32)
        state["used"] += int(n.max())
        tokens.append(np.where(np.arange(K + 1)[None, :] < n[:, None], t, -1))
        counts.append(n)
    out = dict(tokens=np.stack(tokens), counts=np.stack(counts), hidden=dec.debug(DBG_H_LAST))
    if case["logits"]:
        out["logits"] = dec.debug(DBG_LOGITS)
    return out


# ---------------------------------------------------------------- what a pass needs
def work(case):
    if case["op"] == "labels":
        return {"bytes": 4 * case["seqs"] * case["length"] * (case["heads"] + 2), "flops": 0}
    if case["op"] == "linear":
        e = 2 if case["dtype"] == "bf16" else 4
        return {"bytes": e * case["k"] * (case["m"] + case["n"]) + 4 * case["m"] * case["n"], "flops": 2 * case["m"] * case["n"] * case["k"]}
    e = 2 if case["dtype"] == "bf16" else 4
    d, F, V, L, K = case["d"], case["ffn"], case["vocab"], case["layers"], len(_caps(case))
    q, kv = case["heads"] * case["hd"], case["kv"] * case["hd"]
    layer = 2 * d * q + 2 * d * kv + 3 * d * F
    n = [case["prompt_hi"]] if case["batch"] == 1 else np.linspace(case["prompt_lo"], case["prompt_hi"], case["batch"])
    total, squares, B, T = float(np.sum(n)), float(np.sum(np.square(n))), case["batch"], case["nodes"]
    by = fl = 0.0
    if case["op"] != "decode":
        by += e * (L * layer + V * d + total * d + L * 2 * kv * total)
        fl += 2 * total * L * layer + 2 * B * V * d + 2 * L * q * squares
    if case["op"] != "prefill":
        heads = K * (d * d + d) + V * d
        by += case["steps"] * e * (L * layer + V * d + heads + B * T * d + L * 2 * kv * (total + B * T))
        fl += case["steps"] * (2 * B * T * (L * layer + V * d) + 2 * B * K * (d * d + V * d) + 4 * L * q * T * total)
        if case["logits"]:
            by += 4 * B * T * V
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """Measured against another order of the sums and against `exact`, times about four."""
    if case["op"] == "labels":
        return "exact"
    if case["op"] == "linear":
        return {"rel": 1e-5 if case["dtype"] == "fp32" else 2e-5, "max": 4e-4}
    if case["dtype"] == "fp32":
        return {"rel": 2e-5, "max": 4e-4}
    # bf16 operands: a rounding that falls the other way in one layer travels through those that follow
    return {"rel": 0.02, "max": 0.2}


# ---------------------------------------------------------------- the same in 64 bits, plain torch
def exact(case, seed):
    if case["op"] == "labels":
        return None
    if case["op"] == "linear":
        s = prepare(case, seed)
        return s["x"].double() @ s["w"].double().T
    return _Exact(case, seed).run()


class _Exact:
    def __init__(self, case, seed):
        self.c, self.w, self.prompts = case, _weights(case, seed), _prompts(case, seed)
        self.tables = _tables(case, seed, self.prompts)
        paths = [()]
        caps = _caps(case)
        level = [()]
        for cap in caps:
            level = [p + (r,) for p in level for r in range(cap)]
            paths += level
        paths = [()] + sorted(paths[1:], key=lambda p: (sum(p) + len(p), len(p), p))[:case["nodes"] - 1]
        at = {p: i for i, p in enumerate(paths)}
        self.paths = paths
        self.parent = [-1] + [at[p[:-1]] for p in paths[1:]]
        T = len(paths)
        self.sees = torch.zeros((T, T), dtype=torch.bool, device=DEVICE)
        for v in range(T):
            u = v
            while u >= 0:
                self.sees[v, u] = True
                u = self.parent[u]
        D = case["hd"]
        base = 1e6 if case["dtype"] == "bf16" else 1e4
        self.inv = torch.tensor([base ** (-2.0 * i / D) for i in range(D // 2)], dtype=torch.float64, device=DEVICE)

    def norm(self, x, g):
        return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + 1e-5) * g.double()

    def rope(self, x, pos):
        a = pos.double()[:, None, None] * self.inv
        h = x.shape[-1] // 2
        x1, x2 = x[..., :h], x[..., h:]
        return torch.cat([x1 * a.cos() - x2 * a.sin(), x2 * a.cos() + x1 * a.sin()], -1)

    def forward(self, tokens, pos, cache, sees):
        """Rows after the cached ones (cache: per layer (k, v) or empty). Returns hidden rows and the rows' new (k, v)."""
        c, w = self.c, self.w
        H, KV, D, R = c["heads"], c["kv"], c["hd"], len(tokens)
        x = w["embed"][tokens].double()
        new = []
        for l in range(c["layers"]):
            p = f"layers.{l}."
            qkv = self.norm(x, w[p + "attn_norm"]) @ w[p + "wqkv"].double().T
            q = self.rope(qkv[:, :H * D].view(R, H, D), pos)
            k = self.rope(qkv[:, H * D:(H + KV) * D].view(R, KV, D), pos)
            v = qkv[:, (H + KV) * D:].view(R, KV, D)
            new.append((k, v))
            n = cache[l][0].shape[0] if cache else 0
            ka, va = (torch.cat([cache[l][0], k]), torch.cat([cache[l][1], v])) if n else (k, v)
            o = torch.empty((R, H, D), dtype=torch.float64, device=DEVICE)
            for h in range(H):
                s = q[:, h] @ ka[:, h * KV // H].T / math.sqrt(D)
                s[:, n:].masked_fill_(~sees, -math.inf)
                o[:, h] = torch.softmax(s, -1) @ va[:, h * KV // H]
            x = x + o.view(R, H * D) @ w[p + "wo"].double().T
            u = self.norm(x, w[p + "ffn_norm"])
            a = torch.nn.functional.silu(u @ w[p + "w_gate"].double().T) * (u @ w[p + "w_up"].double().T)
            x = x + a @ w[p + "w_down"].double().T
        return self.norm(x, w["final_norm"]), new

    def run(self):
        c = self.c
        K, steps = len(_caps(c)), c["steps"]
        lm = self.w["lm_head"].double()
        tokens = np.full((steps, c["batch"], K + 1), -1, dtype=np.int32)
        counts = np.zeros((steps, c["batch"]), dtype=np.int32)
        hidden, first, logits = [], [], []
        kmax = _kmax(c)
        for b, prompt in enumerate(self.prompts):
            n = len(prompt)
            t = torch.from_numpy(prompt.astype(np.int64)).to(DEVICE)
            causal = torch.ones((n, n), dtype=torch.bool, device=DEVICE).tril_()
            h, cache = self.forward(t, torch.arange(n, device=DEVICE), None, causal)
            h = h[-1]
            root = int((lm @ h).argmax())
            first.append(root)
            for k in range(steps if c["op"] != "prefill" else 0):
                z = []
                for i in range(K):
                    r = h + torch.nn.functional.silu(self.w[f"medusa.{i}.w"].double() @ h + self.w[f"medusa.{i}.b"].double())
                    z.append((lm @ r).topk(kmax).indices.tolist())
                if self.tables is not None:
                    roots = np.full(c["batch"], root, dtype=np.int32)
                    z = _override(c, self.tables, k, roots)[b].tolist()
                tok = torch.tensor([root] + [z[len(p) - 1][p[-1]] for p in self.paths[1:]], device=DEVICE)
                pos = torch.tensor([n + len(p) for p in self.paths], device=DEVICE)
                hid, new = self.forward(tok, pos, cache, self.sees)
                zz = hid @ lm.T
                best = zz.argmax(-1).tolist()
                if c["temperature"] > 0:
                    pr = torch.softmax(zz / c["temperature"], -1)
                    limit = torch.clamp(TYP_DELTA * torch.exp((pr * torch.log(pr.clamp_min(1e-300))).sum(-1)), max=TYP_EPS)
                ok, at = [True], 0
                for v in range(1, len(self.paths)):
                    u = self.parent[v]
                    fits = int(tok[v]) == best[u] if c["temperature"] <= 0 else bool(pr[u, tok[v]] > limit[u])
                    ok.append(ok[u] and fits)
                    if ok[v] and len(self.paths[v]) > len(self.paths[at]):
                        at = v
                path, v = [], at
                while v >= 0:
                    path.insert(0, v)
                    v = self.parent[v]
                keep = torch.tensor(path, device=DEVICE)
                cache = [(torch.cat([ck, nk[keep]]), torch.cat([cv, nv[keep]])) for (ck, cv), (nk, nv) in zip(cache, new)]
                tokens[k, b, :len(path)] = tok[keep].cpu().numpy()
                counts[k, b] = len(path)
                n += len(path)
                # (sampled decoding draws here; with this model's peaked distribution the draw is the largest)
                h, root = hid[at], best[at]
            hidden.append(h)
            if c["logits"]:
                logits.append(zz)
            del cache
        if c["op"] == "prefill":
            return dict(next=np.array(first, dtype=np.int32), hidden=torch.stack(hidden))
        out = dict(tokens=tokens, counts=counts, hidden=torch.stack(hidden))
        if c["logits"]:
            out["logits"] = torch.cat(logits)
        return out
