"""The work that a program using this drafter has it do, as cases that can be timed and compared.

A pass is one draft round through the ``Drafter`` (or the LM-head entry point for callers
that cannot allocate), followed by the acceptance call that ends it, as a serving loop makes
them.  Shapes are those of this repository's workloads and tests.  Contexts are sized as the
README's example sizes them: ``max_new = K + 1``, the most tokens a round can accept, and
every sequence brings between 1 and K + 1 of them, as the previous round's acceptance left it.

Inputs come from the seed alone.  Weights are normal, with gains of a trained layer's order,
and the LM head gives each token a few likely successors: its row for successor r of token x
holds a multiple w_r of E(x).  Drafts are then decided by clear margins, as a trained
drafter's are, so the tokens of a chain do not hang on the last bit of a logit.
"""
import math

import torch

from paper_2602_01762_gb300 import Drafter, lm_head_topk_static

EPS = 1e-5
SHAPES = {
    "tiny": dict(hidden=256, n_q_heads=4, n_kv_heads=4, head_dim=64, ffn=688, vocab=4096, n_steps=3, rope_theta=1e4),
    "mid": dict(hidden=1024, n_q_heads=8, n_kv_heads=2, head_dim=128, ffn=2816, vocab=32000, n_steps=4, rope_theta=1e4),
    "llama3-8b": dict(hidden=4096, n_q_heads=32, n_kv_heads=8, head_dim=128, ffn=14336, vocab=128256, n_steps=5,
                      rope_theta=5e5),
    "llama2-7b": dict(hidden=4096, n_q_heads=32, n_kv_heads=32, head_dim=128, ffn=11008, vocab=32000, n_steps=7,
                      rope_theta=1e4),
    "llama3-70b": dict(hidden=8192, n_q_heads=64, n_kv_heads=8, head_dim=128, ffn=28672, vocab=128256, n_steps=5,
                       rope_theta=5e5),
}
# successors' strengths: the first clearly ahead, the others graded (top-k lists, tree branches)
STRENGTH = (1.5, 0.95, 0.85, 0.75, 0.66, 0.58, 0.5, 0.43)


def _round(name, mode, shape, batch, ctx, *, dtype="bf16", new=None, topk=1, logits=False, steps=0, vocab=0, width=0,
           nodes=0):
    """One round's case: ``ctx`` and ``new`` are the (least, most) committed rows and tokens fed to step 1."""
    k = steps or SHAPES[shape]["n_steps"]
    lo, hi = new or (1, k + 1)
    case = {"name": name, "mode": mode, "shape": shape, "dtype": dtype, "batch": batch, "ctx_lo": ctx[0],
            "ctx_hi": ctx[1], "new_lo": lo, "new_hi": hi, "topk": topk, "logits": logits, "steps": k,
            "vocab": vocab or SHAPES[shape]["vocab"], "width": width, "nodes": nodes}
    return {k: v for k, v in case.items() if k != "name" or v}


def _head(name, shape, rows, *, dtype="bf16", topk=8, vocab=0, norm=True):
    case = {"name": name, "mode": "head", "shape": shape, "dtype": dtype, "batch": rows, "topk": topk, "norm": norm,
            "vocab": vocab or SHAPES[shape]["vocab"]}
    return {k: v for k, v in case.items() if k != "name" or v}


def listed():
    return [
        # a small drafter on one sequence: weights stay in L2, latency and launches count
        _round("tiny-b1", "chain", "tiny", 1, (64, 64), logits=True),
        # 32-bit weights, a few ragged sequences
        _round("mid-f32-b3", "chain", "mid", 3, (40, 200), dtype="f32", topk=4, logits=True),
        # one user at a time: the interactive round, every weight read once per step
        _round("8b-b1", "chain", "llama3-8b", 1, (2048, 2048), logits=True),
        # small batch, many steps, as many KV heads as query heads
        _round("7b-b8", "chain", "llama2-7b", 8, (1024, 1024)),
        # a server's ordinary batch with candidate lists and contexts of uneven length
        _round("8b-b16-top8", "chain", "llama3-8b", 16, (512, 4096), topk=8),
        # the same server under load
        _round("8b-b64-top8", "chain", "llama3-8b", 64, (512, 4096), topk=8),
        # the largest drafter
        _round("70b-b32", "chain", "llama3-70b", 32, (4096, 4096)),
        # a request's first round: its prompt goes through step 1 into an empty draft cache
        _round("8b-prompt-1000", "chain", "llama3-8b", 1, (0, 0), new=(1000, 1000), logits=True),
        # sampled drafting with speculative-sampling acceptance
        _round("8b-sampled-b8", "sampled", "llama3-8b", 8, (512, 2048), logits=True),
        # the paper's tree: 6 steps, 4 branches, 16 verified nodes
        _round("8b-tree-b1", "tree", "llama3-8b", 1, (2048, 2048), logits=True, steps=6, width=4, nodes=16),
        # a shallower tree for a few users at a time
        _round("8b-tree-b4", "tree", "llama3-8b", 4, (512, 2048), steps=4, width=4, nodes=12),
        # the LM head alone, for a host that owns all device memory
        _head("8b-head-b16", "llama3-8b", 16),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("small", "chain", "chain", "large", "prompt", "sampled", "tree", "head"))
    big = rng.choice(("llama3-8b", "llama3-8b", "llama2-7b"))
    c0 = _log(rng, 32, 3000)
    ctx = (c0, rng.randint(c0, 4096))
    if kind == "small":
        dtype = rng.choice(("f32", "bf16"))
        shape = rng.choice(("tiny", "mid"))
        return _round("", "chain", shape, _log(rng, 1, 24), (min(c0, 400), min(ctx[1], 600)), dtype=dtype,
                      topk=rng.choice((1, 3, 8)), logits=True, vocab=rng.choice((0, 4000 + rng.randint(0, 90))))
    if kind == "chain":
        return _round("", "chain", big, _log(rng, 1, 64), ctx, topk=rng.choice((1, 1, 5, 8)))
    if kind == "large":
        return _round("", "chain", "llama3-70b", _log(rng, 4, 32), ctx, topk=1)
    if kind == "prompt":
        batch = rng.choice((1, 1, 2, 4))
        hi = _log(rng, 48, 2000 // batch)
        return _round("", "chain", rng.choice((big, "mid")), batch, (0, 0), new=(rng.randint(hi // 2, hi), hi),
                      logits=True)
    if kind == "sampled":
        return _round("", "sampled", rng.choice((big, "mid")), _log(rng, 1, 16), ctx, logits=True)
    if kind == "tree":
        width, steps = rng.randint(2, 6), rng.randint(3, 6)
        return _round("", "tree", rng.choice((big, "mid")), _log(rng, 1, 6), ctx, steps=steps, width=width,
                      nodes=rng.randint(6, min(16, width + (steps - 1) * width * width)))
    dtype = rng.choice(("bf16", "bf16", "bf16", "f32"))
    return _head("", rng.choice(("mid", big)), _log(rng, 1, 64), dtype=dtype, topk=rng.randint(1, 8),
                 norm=rng.random() < 0.7, vocab=rng.choice((0, rng.randint(9000, 60000))))


# ------------------------------------------------------------------------------------------ inputs


def _width(case):
    return case.get("width", 0)


def _max_ctx(case):
    tail = max(case["steps"], (case["steps"] - 1) * _width(case))
    return (case["ctx_hi"] + case["new_hi"] + tail + 15) // 16 * 16


def _successors(g, vocab, d, n, dtype, dev, branch=None):
    """Embedding, LM head and the n successors of every token (in order of strength).  ``branch``: the tokens after
    which the others than the first are likely too (None: after every token)."""
    embed = torch.randn(vocab, d, generator=g, device=dev, dtype=dtype) * 0.5
    head = torch.randn(vocab, d, generator=g, device=dev, dtype=dtype) * (0.2 / math.sqrt(d))
    amp = torch.exp(0.15 * torch.randn(vocab, generator=g, device=dev))
    rest = torch.ones(vocab, device=dev)
    if branch is not None:
        rest.fill_(0.3).index_fill_(0, branch, 1.0)
    succ = []
    for r in range(n):
        perm = torch.randperm(vocab, generator=g, device=dev)
        succ.append(perm)
        back = torch.empty_like(perm)
        back[perm] = torch.arange(vocab, device=dev)
        coef = (STRENGTH[r] * 40.0 / d * (amp * rest if r else amp)[back]).to(dtype)
        for i in range(0, vocab, 16384):
            head[i:i + 16384].addcmul_(embed[back[i:i + 16384]], coef[i:i + 16384, None])
    return embed, head, succ


def _module(g, s, dtype, dev):
    d, f, hd = s["hidden"], s["ffn"], s["head_dim"]
    q = s["n_q_heads"] * hd
    qkv = q + 2 * s["n_kv_heads"] * hd

    def w(rows, kin, gain):
        return torch.randn(rows, kin, generator=g, device=dev, dtype=dtype).mul_(gain / math.sqrt(kin))

    def gain():
        return (1 + 0.1 * torch.randn(d, generator=g, device=dev)).to(dtype)

    # the fusion passes the token on (identity plus noise) beside the mixed hidden state
    fuse = torch.cat([w(d, d, 0.4) + torch.eye(d, device=dev, dtype=dtype), w(d, d, 0.3)], 1).contiguous()
    return {"w_fuse": fuse, "g_attn": gain(), "w_qkv": w(qkv, d, 1.2), "w_o": w(d, q, 1.2), "g_mlp": gain(),
            "w_gate_up": w(2 * f, d, 1.2), "w_down": w(d, f, 0.5), "g_final": gain()}


def _data(case, seed):
    """Weights and inputs of a case, from the seed alone."""
    dev = torch.device("cuda", torch.cuda.current_device())
    g = torch.Generator(device=dev).manual_seed(seed)
    h = torch.Generator().manual_seed(seed)
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    s = dict(SHAPES[case["shape"]], vocab=case["vocab"])
    b, d, v = case["batch"], s["hidden"], s["vocab"]
    x = {"shape": s, "dtype": dtype, "dev": dev}
    if case["mode"] == "head":
        # hidden rows whose best tokens are graded like the successors above
        x["lm_head"] = torch.randn(v, d, generator=g, device=dev, dtype=dtype) * (1.2 / math.sqrt(d))
        pick = torch.randint(0, v, (b, 8), generator=h).to(dev)
        mix = torch.tensor(STRENGTH, device=dev) * (1 + 0.1 * torch.rand(b, 8, generator=g, device=dev))
        x["h"] = (torch.einsum("br,brd->bd", mix, x["lm_head"][pick].float()) * 15
                  + 0.5 * torch.randn(b, d, generator=g, device=dev)).contiguous()
        x["g_final"] = (1 + 0.1 * torch.randn(d, generator=g, device=dev)).to(dtype) if case["norm"] else None
        return x
    k, n_max, w = case["steps"], case["new_hi"], _width(case)
    n_succ = max(case["topk"], w, 2)
    x["tokens"] = torch.randint(0, v, (b, n_max), generator=h).to(torch.int32)
    x["n_new"] = torch.randint(case["new_lo"], n_max + 1, (b,), generator=h).to(torch.int32)
    last = x["tokens"].gather(1, x["n_new"].long()[:, None] - 1)[:, 0].to(dev).long()
    # a tree's paths are ranked by sums of log-probabilities: the text branches after the last accepted token and is
    # sure of itself from there on, so that no two sums are nearly the same
    x["embed"], x["lm_head"], succ = _successors(g, v, d, n_succ, dtype, dev, last if w else None)
    x["modules"] = [_module(g, s, dtype, dev) for _ in range(k)]
    x["kv_len"] = torch.randint(case["ctx_lo"], case["ctx_hi"] + 1, (b,), generator=h).to(torch.int32)
    x["hidden"] = torch.randn(b, n_max, d, generator=g, device=dev, dtype=dtype)
    cache = (b, s["n_kv_heads"], _max_ctx(case), s["head_dim"])
    x["k_cache"] = torch.randn(cache, generator=g, device=dev, dtype=dtype)
    x["v_cache"] = torch.randn(cache, generator=g, device=dev, dtype=dtype)
    # the target agrees with the likely chain for a while, then takes a token of its own
    chain = []
    for _ in range(k + 1):
        last = succ[0][last]
        chain.append(last)
    agree = torch.randint(0, k + 1, (b, 1), generator=h)
    other = torch.randint(0, v, (b, k + 1), generator=h)
    target = torch.where(torch.arange(k + 1)[None] < agree, torch.stack(chain, 1).cpu(), other)
    if case["mode"] == "sampled":
        sure = 0.9995           # a draw from the flat rest would hang on the last bits of its running sum
        p = torch.randn(b, k + 1, v, generator=g, device=dev).softmax(-1).mul_(1 - sure)
        x["target_probs"] = p.scatter_add_(2, target.to(dev)[:, :, None], torch.full((b, k + 1, 1), sure, device=dev))
        x["seed"] = torch.randint(1, 1 << 62, (1,), generator=h)
    if case["mode"] == "tree":
        # the target's token after each node: the likely successor of some, its own after others
        x["target_next"] = torch.randint(0, v, (b, case["nodes"] + 1), generator=h).to(torch.int32)
        x["target_next"][:, 0] = chain[0].cpu().to(torch.int32)
    x["target"] = target.to(torch.int32)
    return x


def prepare(case, seed):
    x = _data(case, seed)
    dev, s = x["dev"], x["shape"]
    b, f32, i32 = case["batch"], torch.float32, torch.int32

    def out(*shape, dtype=f32):
        return torch.zeros(shape, dtype=dtype, device=dev)

    if case["mode"] == "head":
        x["out"] = {"draft": out(b, dtype=i32), "topk_ids": out(b, case["topk"], dtype=i32),
                    "topk_logits": out(b, case["topk"]), "logits": out(b, s["vocab"])}
        return {"case": case, "x": x}
    k, w, n = case["steps"], _width(case), case["nodes"]
    dr = Drafter(**{**s, "n_steps": k}, dtype=case["dtype"], max_batch=b, max_ctx=_max_ctx(case), max_new=case["new_hi"],
                 topk=case["topk"], rms_eps=EPS, max_tree_width=w, device=dev.index)
    dr.load_shared_weights(x["embed"], x["lm_head"])
    for i, m in enumerate(x["modules"]):
        dr.load_step_weights(i, m)
    for name in ("tokens", "n_new", "kv_len", "target", "target_next", "seed"):
        if name in x:
            x[name] = x[name].to(dev)
    o = {"accept_len": out(b, dtype=i32), "out_tokens": out(b, k + 1, dtype=i32), "kv_len": x["kv_len"].clone()}
    if case["mode"] == "tree":
        o.update(tokens=out(b, n, dtype=i32), parents=out(b, n, dtype=i32), depths=out(b, n, dtype=i32), scores=out(b, n),
                 frontier=out(b, k, w, dtype=i32), accept_nodes=out(b, k, dtype=i32))
        if case["logits"]:
            o["row_logits"] = out(k, b, w, s["vocab"])
    else:
        o.update(draft_ids=out(b, k, dtype=i32), topk_ids=out(b, k, case["topk"], dtype=i32),
                 topk_logits=out(b, k, case["topk"]), hidden=out(b, k, s["hidden"]))
        if case["logits"]:
            o["logits"] = out(b, k, s["vocab"])
        if case["mode"] == "sampled":
            o["lse"] = out(b, k)
    x["out"] = o
    return {"case": case, "x": x, "drafter": dr}


def run(state):
    case, x = state["case"], state["x"]
    o = x["out"]
    if case["mode"] == "head":
        lm_head_topk_static(x["h"], x["g_final"], x["lm_head"], o["draft"], o["topk_ids"], o["topk_logits"], o["logits"],
                            rms_eps=EPS)
        return dict(o)
    dr = state["drafter"]
    o["kv_len"].copy_(x["kv_len"])              # the round's committed lengths; the acceptance advances them
    head = (x["tokens"], x["hidden"], x["n_new"], o["kv_len"], x["k_cache"], x["v_cache"])
    if case["mode"] == "tree":
        dr.draft_tree(*head, case["width"], o["tokens"], o["parents"], o["depths"], o["scores"], frontier=o["frontier"],
                      row_logits=o.get("row_logits"))
        dr.accept_tree(o["tokens"], o["parents"], x["target_next"], x["n_new"], o["kv_len"], o["accept_len"],
                       o["accept_nodes"], o["out_tokens"])
    elif case["mode"] == "sampled":
        dr.draft_round_sampled(*head, 1.0, x["seed"], o["draft_ids"], o["logits"], o["lse"], topk_ids=o["topk_ids"],
                               topk_logits=o["topk_logits"], hidden_out=o["hidden"])
        dr.accept_sampled(o["draft_ids"], o["logits"], o["lse"], 1.0, x["target_probs"], x["seed"], x["n_new"],
                          o["kv_len"], o["accept_len"], o["out_tokens"])
    else:
        dr.draft_round(*head, o["draft_ids"], o["topk_ids"], o["topk_logits"], o.get("logits"), o["hidden"])
        dr.accept_greedy(o["draft_ids"], x["target"], x["n_new"], o["kv_len"], o["accept_len"], o["out_tokens"])
    return dict(o, k_cache=x["k_cache"], v_cache=x["v_cache"])


# ------------------------------------------------------------------------------------------ what it needs


def work(case):
    s = SHAPES[case["shape"]]
    d, f, v, b = s["hidden"], s["ffn"], case["vocab"], case["batch"]
    es = 2 if case["dtype"] == "bf16" else 4
    if case["mode"] == "head":
        return {"bytes": v * d * es + b * (d + v + 2 * case["topk"]) * 4, "flops": 2 * b * v * d}
    q, kv = s["n_q_heads"] * s["head_dim"], s["n_kv_heads"] * s["head_dim"]
    k, w = case["steps"], max(_width(case), 1)
    new, ctx = (case["new_lo"] + case["new_hi"]) / 2, (case["ctx_lo"] + case["ctx_hi"]) / 2
    fuse, wkv, wq, mlp = 2 * d * d, 2 * kv * d, q * d, d * q + 3 * d * f
    weights = k * (fuse + wkv + wq + mlp + v * d + 3 * d)
    rows = b * (1 + (k - 1) * w)                                # rows that go through a whole layer and the LM head
    macs = b * new * (fuse + wkv) + b * (wq + mlp + v * d) + (rows - b) * (fuse + wkv + wq + mlp + v * d)
    seen = b * sum(ctx + new + i * w for i in range(k))         # cache rows read, once per step
    macs += 2 * (b * (ctx + new) + (rows - b) * (ctx + new + k * w / 2)) * q
    moved = seen * 2 * kv + (b * new + rows - b) * 2 * kv + (b * new + rows) * d + b * new * d
    outs = rows * (v if case["logits"] else 0) + (rows * d if case["mode"] != "tree" else 0)
    if case["mode"] == "sampled":
        outs += b * (k + 1) * v                                 # the target's probabilities
    return {"bytes": (weights + moved) * es + outs * 4, "flops": 2 * macs}


def tolerance(case):
    # about four times what the tensor-core kernels differ from the CUDA-core ones on these cases: each bf16 operand
    # that rounds the other way travels through the steps that follow; the head alone rounds one row; 32 bits round sums
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.002}
    if case["mode"] == "head":
        return {"rel": 2e-3, "max": 0.02, "differ": 0.01}
    return {"rel": 0.02, "max": 0.2, "differ": 0.01}


# ------------------------------------------------------------------------------------------ in 64 bits


def _mm(x, w):
    return torch.cat([x @ w[i:i + 4096].double().T for i in range(0, w.shape[0], 4096)], 1)


def _norm(x, gain):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + EPS) * gain.double()


def _rope(x, pos, theta):
    half = x.shape[-1] // 2
    a = pos.double()[:, None] * theta ** (-torch.arange(half, device=x.device, dtype=torch.float64) / half)
    c, s = a.cos()[:, None], a.sin()[:, None]
    return torch.cat([x[..., :half] * c - x[..., half:] * s, x[..., half:] * c + x[..., :half] * s], -1)


def _layer(x, m, u, pos, slot, seq, cache, queries, visible):
    """Rows u [T, 2d] of sequences ``seq`` through one module; K/V of each row are stored at its slot.  The rows
    ``queries`` attend to the cache rows visible(row) and go on; their hidden rows are returned."""
    s = x["shape"]
    hd, nq, nk = s["head_dim"], s["n_q_heads"], s["n_kv_heads"]
    x0 = _mm(u, m["w_fuse"])
    n1 = _norm(x0, m["g_attn"])
    kv = _mm(n1, m["w_qkv"][nq * hd:]).view(-1, 2 * nk, hd)
    cache[0][seq, :, slot] = _rope(kv[:, :nk], pos, s["rope_theta"])
    cache[1][seq, :, slot] = kv[:, nk:]
    q = _rope(_mm(n1[queries], m["w_qkv"][:nq * hd]).view(-1, nq, hd), pos[queries], s["rope_theta"])
    o = torch.empty(len(queries), nq * hd, dtype=torch.float64, device=u.device)
    for i, r in enumerate(queries.tolist()):
        b = int(seq[r])
        rows = visible(r)
        kk, vv = cache[0][b][:, rows], cache[1][b][:, rows]
        p = torch.einsum("hgd,hnd->hgn", q[i].view(nk, -1, hd), kk).div(math.sqrt(hd)).softmax(-1)
        o[i] = torch.einsum("hgn,hnd->hgd", p, vv).reshape(-1)
    a = x0[queries] + _mm(o, m["w_o"])
    n2 = _norm(a, m["g_mlp"])
    f = s["ffn"]
    gate = _mm(n2, m["w_gate_up"][:f])
    return a + _mm(torch.nn.functional.silu(gate) * _mm(n2, m["w_gate_up"][f:]), m["w_down"])


def _wrap(v):
    """An unsigned 64-bit constant as the signed value of the same bits."""
    return v - (1 << 64) if v >= 1 << 63 else v


def _gumbel(seed, b, k, vocab, dev):
    """Gumbel noise of the draft draw: the SplitMix64 counter stream that the header describes."""
    def shr(z, n):
        return (z >> n) & ((1 << (64 - n)) - 1)
    n = torch.arange(vocab, device=dev, dtype=torch.int64) + ((1 << 60) | (b << 40) | (k << 32)) + 1
    z = n * _wrap(0x9E3779B97F4A7C15) + int(seed)
    z = (z ^ shr(z, 30)) * _wrap(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * _wrap(0x94D049BB133111EB)
    u = (shr(z ^ shr(z, 31), 41).double() + 0.5) / 8388608
    return -torch.log(-torch.log(u))


def exact(case, seed):
    x = _data(case, seed)
    s, dev = x["shape"], x["dev"]
    b, v = case["batch"], s["vocab"]
    if case["mode"] == "head":
        h = x["h"].double()
        z = _mm(h if x["g_final"] is None else _norm(h, x["g_final"]), x["lm_head"])
        return {"draft": None, "topk_ids": None, "topk_logits": z.topk(case["topk"]).values, "logits": z}
    k_steps, w, kn = case["steps"], _width(case), case["topk"]
    kv, new = x["kv_len"].long(), x["n_new"].long()
    cache = [x.pop("k_cache").double(), x.pop("v_cache").double()]
    first = [(i, j) for i in range(b) for j in range(int(new[i]))]
    seq = torch.tensor([p[0] for p in first])
    at = torch.tensor([p[1] for p in first])
    ends = torch.cumsum(new, 0) - 1
    tok = x["tokens"][seq, at].long().to(dev)
    u = torch.cat([x["embed"][tok], x["hidden"][seq.to(dev), at.to(dev)]], 1).double()
    pos = (kv[seq] + at).to(dev)
    base = (kv + new).tolist()
    h = _layer(x, x["modules"][0], u, pos, pos, seq.to(dev), cache, ends.to(dev),
               lambda r: slice(0, int(pos[r]) + 1))
    o = {"accept_len": None, "out_tokens": None, "kv_len": None}
    every = torch.arange(b, device=dev)
    hidden, logits, lse, top = [], [], [], []
    if case["mode"] != "tree":
        for k in range(1, k_steps + 1):
            m = x["modules"][k - 1]
            if k > 1:
                slots = torch.tensor([n + k - 2 for n in base], device=dev)
                h = _layer(x, m, torch.cat([x["embed"][nxt].double(), h], 1), slots, slots, every, cache, every,
                           lambda r: slice(0, base[r] + k - 1))
            z = _mm(_norm(h, m["g_final"]), x["lm_head"])
            hidden.append(h)
            logits.append(z if case["logits"] else None)
            lse.append(z.logsumexp(-1))
            top.append(z.topk(kn).values)
            nxt = z.argmax(-1)
            if case["mode"] == "sampled":
                nxt = torch.stack([(z[i] + _gumbel(x["seed"], i, k - 1, v, dev)).argmax() for i in range(b)])
        o.update(draft_ids=None, topk_ids=None, topk_logits=torch.stack(top, 1), hidden=torch.stack(hidden, 1))
        if case["logits"]:
            o["logits"] = torch.stack(logits, 1)
        if case["mode"] == "sampled":
            o["lse"] = torch.stack(lse, 1)
        return dict(o, k_cache=cache[0], v_cache=cache[1])
    # tree: the w best of each row are candidates, the w best candidates of a step its frontier
    n = case["nodes"]
    row_logits = torch.zeros(k_steps, b, w, v, dtype=torch.float64, device=dev) if case["logits"] else None
    pool = [[] for _ in range(b)]                                # per sequence: (score, token, row that proposed it)
    front = [[] for _ in range(b)]
    slots_of = [{(1, 0): []} for _ in range(b)]                  # per row: cache slots of it and its ancestors
    hid = [{} for _ in range(b)]
    for k in range(1, k_steps + 1):
        m = x["modules"][k - 1]
        if k == 1:
            names = [(i, 0) for i in range(b)]
        else:
            names = [(i, j) for i in range(b) for j in range(w)]
            for i, j in names:
                slots_of[i][(k, j)] = slots_of[i][pool[i][front[i][j]][2]] + [base[i] + (k - 2) * w + j]
            u = torch.stack([torch.cat([x["embed"][pool[i][front[i][j]][1]].double(), hid[i][pool[i][front[i][j]][2]]])
                             for i, j in names])
            sq = torch.tensor([i for i, _ in names], device=dev)
            ps = torch.tensor([base[i] + k - 2 for i, _ in names], device=dev)
            sl = torch.tensor([slots_of[i][(k, j)][-1] for i, j in names], device=dev)

            def visible(r):
                i, j = names[r]
                return torch.tensor(list(range(base[i])) + slots_of[i][(k, j)], device=dev)
            h = _layer(x, m, u, ps, sl, sq, cache, torch.arange(len(names), device=dev), visible)
        z = _mm(_norm(h, m["g_final"]), x["lm_head"])
        best, ids = z.topk(w)
        lp = (best - z.logsumexp(-1, keepdim=True)).tolist()
        ids = ids.tolist()
        start = [len(p) for p in pool]
        for r, (i, j) in enumerate(names):
            hid[i][(k, j)] = h[r]
            if case["logits"]:
                row_logits[k - 1, i, j] = z[r]
            above = pool[i][front[i][j]][0] if k > 1 else 0.0
            pool[i] += [(above + lp[r][c], ids[r][c], (k, j)) for c in range(w)]
        front = [sorted(range(start[i], len(pool[i])), key=lambda e: (-pool[i][e][0], e))[:w] for i in range(b)]
    chosen = [sorted(sorted(range(len(p)), key=lambda e: (-p[e][0], e))[:n]) for p in pool]
    o.update(tokens=None, parents=None, depths=None, frontier=None, accept_nodes=None,
             scores=torch.tensor([[p[e][0] for e in c] for p, c in zip(pool, chosen)], dtype=torch.float64))
    if case["logits"]:
        o["row_logits"] = row_logits
    return dict(o, k_cache=cache[0], v_cache=cache[1])
