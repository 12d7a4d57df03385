"""The work that users of this library have it do, as timed cases: decode steps, autoregressive steps and prompts.

A case names a model shape (`synth.CONFIGS`, at its own or a reduced depth; `small` is the bf16 model of the test suite),
a batch with its context lengths, and the beam.  Weights are random with three properties of a trained model that plain
random weights lack and that decide what a step does:

* embeddings of unit size and residual projections scaled by 1/sqrt(2 layers), the usual initialisation of a deep
  network, so that depth does not drown the input;
* a language model that is sure of its next token: the output row of the successor of token t points along t's embedding,
  with the same distribution of entries as every other row.  Drafted tokens are then accepted or rejected for a reason,
  contexts grow by several tokens a step, and compaction has rows to move;
* a drafter that knows the same successors.

The greedy stream is therefore known from the seed, and the candidates that a step verifies (`synth.plant_beams`: the
stream with tokens replaced at p = 0.3) can be laid out beforehand for several steps in a row, as can the number of rows
that each step packs.
"""
import math

import numpy as np
import torch

from paper_2403_09919_b200 import binding, synth

# the bf16 model of the test suite: odd tile counts everywhere
SMALL = dict(synth.CONFIGS["tiny"], dtype="bf16", d_model=512, n_heads=4, d_ffn=1376, vocab=1000, d_rnn=512)
PLANT_P, PLANT_RHO = 0.3, 0.5


def _case(name, kind, model, layers, batch, ctx, bw, bl, steps, temperature=0.0):
    return dict(name=name, kind=kind, model=model, layers=layers, batch=batch, ctx_lo=ctx[0], ctx_hi=ctx[1], beam_width=bw,
                beam_length=bl, steps=steps, temperature=temperature)


def listed():
    return [
        # the fp32 configuration: a short burst of steps, all launch latency
        _case("tiny_fp32_steps", "step", "tiny", 2, 1, (64, 64), 4, 4, 8),
        # a small bf16 model: launch latency on the tensor-core path
        _case("small_steps", "step", "small", 4, 2, (90, 160), 8, 5, 4),
        # one user's chat: the headline decode step
        _case("7b_steps", "step", "7b", 32, 1, (512, 512), 8, 5, 2),
        # the same model driven through the four calls of a step, three users, an odd beam
        _case("7b_calls", "calls", "7b", 32, 3, (200, 900), 10, 4, 1),
        # no speculation: autoregressive decoding of a few users
        _case("7b_autoregressive", "ar", "7b", 32, 4, (700, 1500), 8, 5, 4),
        # eight users, sampled output, some 200 rows per verification
        _case("7b_sampled_batch8", "step", "7b", 32, 8, (200, 400), 8, 5, 2, 0.8),
        # a busy server: sixteen users with contexts of very different lengths
        _case("7b_batch16", "step", "7b", 32, 16, (256, 2048), 16, 5, 2),
        # wide beams on one sequence
        _case("13b_wide_beam", "step", "13b", 40, 1, (1024, 1024), 64, 5, 2),
        # long contexts (24 of 60 layers: three copies of the model have to fit the card)
        _case("33b_long_context", "step", "33b", 24, 4, (4096, 4096), 32, 5, 2),
        # prompts: an ordinary one, a ragged batch, a long document
        _case("7b_prompt", "prompt", "7b", 32, 1, (512, 512), 8, 5, 1),
        _case("7b_prompts_ragged", "prompt", "7b", 32, 5, (100, 1700), 8, 5, 1),
        _case("7b_prompt_long", "prompt", "7b", 32, 1, (8192, 8192), 8, 5, 1),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "calls", "ar", "prompt", "prompt"])
    model = rng.choice(["tiny", "small", "7b", "7b", "7b", "13b", "33b"])
    big = model in ("7b", "13b", "33b")
    layers = _log_int(rng, 2, {"tiny": 4, "small": 8, "7b": 32, "13b": 40, "33b": 24}[model])
    batch = _log_int(rng, 1, 16 if model != "33b" else 4)
    bw, bl = _log_int(rng, 1, 64), rng.randint(2, 5)
    if batch * bw > 256:
        bw = max(1, 256 // batch)
    hi = _log_int(rng, 64, 4096 if big else 400)
    lo = hi if rng.random() < 0.3 else rng.randint(max(1, hi // 8), hi)
    steps = rng.randint(1, 3) if big else rng.randint(2, 8)
    temperature = rng.choice([0.0, 0.0, 0.8, 1.0]) if big and kind != "prompt" else 0.0
    c = _case("drawn", kind, model, layers, batch, (lo, hi), bw, bl, 1 if kind in ("calls", "prompt") else steps, temperature)
    if kind == "prompt":
        while c["batch"] > 1 and c["batch"] * c["ctx_hi"] > 8192:   # no more tokens than the longest listed prompt
            c["batch"] -= 1
    largest = max(_seconds(k) for k in listed())
    cfg = _config(c)
    while c["layers"] > 2 and (binding.lib().redrafter_kv_bytes(binding.make_config(cfg)) > 20e9 or _seconds(c) > largest):
        c["layers"] = max(2, c["layers"] * 3 // 4)
        cfg = _config(c)
    del c["name"]
    return c


def _config(case):
    cfg = dict(SMALL if case["model"] == "small" else synth.CONFIGS[case["model"]])
    room = case["steps"] * (1 + case["beam_length"]) + 1 + case["beam_width"] * case["beam_length"]
    cfg.update(n_layers=case["layers"], max_batch=case["batch"], beam_width=case["beam_width"], beam_length=case["beam_length"],
               max_ctx=case["ctx_hi"] + room + 8)
    return cfg


def _plan(case, seed):
    """Everything about a case that is whole numbers: context lengths, the order in which the greedy stream walks the
    vocabulary (one cycle, so it never repeats), roots, and for each step its candidates, how many tokens the model will
    accept, and how many rows the candidates pack to.  Lengths and the candidates' shape, as places along the cycle,
    belong to the case; which tokens these are, to the seed."""
    cfg = _config(case)
    shape = np.random.default_rng([case[k] for k in ("layers", "batch", "ctx_lo", "ctx_hi", "beam_width", "beam_length", "steps")])
    rng = np.random.default_rng(seed)
    B, V, BW, L = case["batch"], cfg["vocab"], case["beam_width"], case["beam_length"]
    order = rng.permutation(V)
    succ = np.empty(V, dtype=np.int64)
    succ[order] = np.roll(order, -1)
    ctx = shape.integers(case["ctx_lo"], case["ctx_hi"] + 1, size=B)
    ctx[shape.integers(0, B)] = case["ctx_hi"]
    place0 = rng.integers(0, V, size=B)
    place, steps = place0.copy(), []
    for _ in range(case["steps"] if case["kind"] in ("step", "calls") else 0):
        beams = np.zeros((B, BW, L), dtype=np.int64)
        took, rows = [], []
        for b in range(B):
            ahead = np.arange(1, L + 1)
            cand = synth.plant_beams(ahead, BW, L, V, shape, p=PLANT_P, rho=PLANT_RHO if BW >= 32 else 0.0)
            took.append(int(max(np.cumprod(cand == ahead, axis=1).sum(axis=1))))
            rows.append(1 + len({tuple(r[:j + 1]) for r in cand.tolist() for j in range(L)}))
            beams[b] = order[(place[b] + cand) % V]
            place[b] = (place[b] + 1 + took[b]) % V
        steps.append(dict(beams=beams, took=took, rows=rows))
    prompts = [rng.integers(0, V, size=int(n)) for n in ctx] if case["kind"] == "prompt" else None
    return dict(cfg=cfg, succ=succ, ctx=ctx, root=order[place0], steps=steps, prompts=prompts)


def _weights(cfg, succ, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    dt = torch.float32 if cfg["dtype"] == "fp32" else torch.bfloat16
    w = {}
    for name, (shape, kind) in synth.weight_shapes(cfg).items():
        t = torch.empty(shape, dtype=dt, device="cuda")
        if kind == "g":
            t.normal_(1.0, 0.05, generator=gen)
        elif name == "tok_emb":
            t.normal_(0.0, 1.0, generator=gen)
        elif name.startswith(("wo.", "w_down.")):
            t.normal_(0.0, 0.02 / math.sqrt(2 * cfg["n_layers"]), generator=gen)
        else:
            t.normal_(0.0, 0.02, generator=gen)
        w[name] = t
    d, nxt = cfg["d_model"], torch.from_numpy(succ).cuda()
    w["lm_head"][nxt] = w["tok_emb"] * 0.02
    # the drafter sees t as E[t] (first call) or through the cell as SiLU(W E[t] + ...): its output row of t's successor
    # points along both
    z = torch.nn.functional.silu((w["tok_emb"] @ w["rnn_w"].t()).float())
    z = (z - z.mean(0)) / z.std(0)
    w["draft_out"][nxt, :d] = (0.02 / math.sqrt(2) * (w["tok_emb"].float() + z)).to(dt)
    return w


def _cache_fill(view, cfg, seed):
    """Keys and values of earlier tokens: what projections of std 0.02 make of a normalised row."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1)
    return view.normal_(0.0, 0.02 * math.sqrt(cfg["d_model"]), generator=gen)


def _hidden(cfg, B, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 2)
    return torch.randn(B, cfg["d_model"], dtype=torch.float32, device="cuda", generator=gen)


def prepare(case, seed):
    p = _plan(case, seed)
    cfg, B = p["cfg"], case["batch"]
    eng = binding.ReDrafter(cfg, _weights(cfg, p["succ"], seed))
    s = dict(eng=eng, case=case, plan=p, ctx_hi=case["ctx_hi"])
    if case["kind"] == "prompt":
        s["prompts"] = [x.astype(np.int32) for x in p["prompts"]]
        return s
    _cache_fill(eng.kv_view(), cfg, seed)
    s["ctx"] = torch.from_numpy(p["ctx"].astype(np.int32)).cuda()
    s["root"] = torch.from_numpy(p["root"].astype(np.int32)).cuda()
    s["h"] = _hidden(cfg, B, seed)
    s["beams"] = [torch.from_numpy(t["beams"].astype(np.int32)).cuda() for t in p["steps"]]
    s["out"] = [binding.AcceptOut(B, case["beam_length"], eng.device) for _ in range(case["steps"])]
    s["token"] = [torch.zeros(B, dtype=torch.int32, device="cuda") for _ in range(case["steps"])]
    s["rows"] = sum(p["steps"][-1]["rows"]) if p["steps"] else B
    if case["temperature"]:
        eng.set_sampling(case["temperature"], seed)
    torch.cuda.synchronize()
    return s


def run(s):
    eng, case = s["eng"], s["case"]
    if case["kind"] == "prompt":
        eng.prefill(s["prompts"])
        ctx, root, h = eng.get_state()
        return dict(ctx=ctx, root=root, hidden=h, logits=eng.last_logits(case["batch"]), kv=eng.kv_view())
    # the batch that a scheduler hands over: contexts, next tokens, hidden states
    eng.set_state(s["ctx"], s["root"], s["h"], batch=case["batch"], ctx_bound=s["ctx_hi"])
    if case["kind"] == "ar":
        for t in s["token"]:
            eng.ar_step(t)
        ctx, root, h = eng.get_state()
        return dict(tokens=s["token"], ctx=ctx, root=root, hidden=h, logits=eng.last_logits(case["batch"]))
    if case["kind"] == "calls":
        drafted, scores = eng.draft()
        packed = eng.pack(s["beams"][0])
        argmax, hidden, logits = eng.verify(packed, want_logits=True)
        out = eng.accept(s["beams"][0], packed, argmax, hidden, s["out"][0])
        ctx, root, h = eng.get_state()
        return dict(drafted=drafted, scores=scores, packed=[packed.tokens, packed.n, packed.unpack, packed.pos, packed.mask,
                    packed.parent], argmax=argmax, rows=hidden, logits=logits,
                    accepted=[out.n_accept, out.best, out.tokens], ctx=ctx, root=root, hidden=h)
    for beams, out in zip(s["beams"], s["out"]):
        eng.step(beams, out)
    ctx, root, h = eng.get_state()
    return dict(accepted=[[o.n_accept, o.best, o.tokens] for o in s["out"]], ctx=ctx, root=root, hidden=h,
                logits=eng.last_logits(s["rows"]))


def _seconds(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / (1.4e15 if case["model"] != "tiny" else 5e13))


def work(case):
    """Weights are read once per forward pass and drafter call (they do not fit on the chip, and each needs the one
    before), cached keys and values once per pass; logits and new keys and values are written."""
    p = _plan(case, 0)
    cfg, B, L = p["cfg"], case["batch"], case["beam_length"]
    d, F, V, dh, n, es = cfg["d_model"], cfg["d_ffn"], cfg["vocab"], 2 * cfg["d_model"], cfg["n_layers"], 4 if cfg["dtype"] == "fp32" else 2
    layers, head = n * (4 * d * d + 3 * d * F), V * d
    kv_row = 2 * d * es * n
    if case["kind"] == "prompt":
        tok = int(p["ctx"].sum())
        att = sum(2.0 * d * n * int(c) * (int(c) + 1) for c in p["ctx"])
        return {"bytes": float((layers + head) * es + tok * (kv_row + d * es + 4) + B * V * 4),
                "flops": 2.0 * tok * layers + 2.0 * B * head + att}
    ctx = int(p["ctx"].sum())
    if case["kind"] == "ar":
        return {"bytes": float(case["steps"] * ((layers + head) * es + (ctx + B) * kv_row + B * V * 4)),
                "flops": case["steps"] * (2.0 * B * (layers + head) + 4.0 * d * n * ctx)}
    drafter = L * (cfg["n_head_layers"] * dh * dh + V * dh) + (L - 1) * 2 * d * d
    drafter_flops = 2.0 * B * ((1 + (L - 1) * case["beam_width"]) * (cfg["n_head_layers"] * dh * dh + V * dh)
                               + (L - 1) * case["beam_width"] * 2 * d * d)
    nbytes = flops = 0.0
    for t in p["steps"]:
        rows = sum(t["rows"])
        nbytes += (layers + head + drafter) * es + (ctx + rows) * kv_row + rows * V * 4
        flops += 2.0 * rows * (layers + head) + drafter_flops + 4.0 * d * n * sum(int(c) * r for c, r in zip(p["ctx"], t["rows"]))
    return {"bytes": float(nbytes), "flops": float(flops)}


def tolerance(case):
    if case["model"] == "tiny":
        return {"rel": 1e-5}
    # bf16 storage between the layers of a deep network, and ranks of drafted candidates that lie within its rounding
    return {"rel": 2e-2, "max": 0.5, "differ": 0.01}


def _norm(x, g, eps):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * g


def _rope(x, pos, theta):
    half = x.shape[-1] // 2
    ang = pos.double()[:, None] * theta ** (-torch.arange(half, dtype=torch.float64, device=x.device) / half)
    c, s = ang.cos()[:, None], ang.sin()[:, None]
    return torch.cat([x[..., :half] * c - x[..., half:] * s, x[..., half:] * c + x[..., :half] * s], -1)


def _forward(w, cfg, seqs, cache=None, keep=None):
    """64-bit forward over the new rows of every sequence.  seqs: dicts of tokens, pos, mask (rows x rows, or None for
    causal) and ctx, the earlier tokens in `cache`.  Returns the rows after the final norm; fills `keep` with K and V."""
    d, H = cfg["d_model"], cfg["n_heads"]
    hd = d // H
    tok = torch.cat([s["tokens"] for s in seqs])
    pos = torch.cat([s["pos"] for s in seqs])
    x = w["tok_emb"][tok].double()
    for l in range(cfg["n_layers"]):
        W = {k: w[f"{k}.{l}"].double() for k in ("attn_norm", "wqkv", "wo", "ffn_norm", "w_gate_up", "w_down")}
        qkv = (_norm(x, W["attn_norm"], cfg["rms_eps"]) @ W["wqkv"].t()).view(-1, 3, H, hd)
        q, k, v = _rope(qkv[:, 0], pos, cfg["rope_theta"]), _rope(qkv[:, 1], pos, cfg["rope_theta"]), qkv[:, 2]
        att, at = torch.empty_like(q), 0
        for b, s in enumerate(seqs):
            n, c = len(s["tokens"]), s["ctx"]
            part = slice(at, at + n)
            at += n
            if keep is not None:
                keep[l, 0, b, :, :n] = k[part].transpose(0, 1)
                keep[l, 1, b, :, :n] = v[part].transpose(0, 1)
            for h in range(H):
                kk, vv = k[part, h], v[part, h]
                if c:
                    kk = torch.cat([cache[l, 0, b, h, :c].double(), kk])
                    vv = torch.cat([cache[l, 1, b, h, :c].double(), vv])
                sc = q[part, h] @ kk.t() / math.sqrt(hd)
                see = s["mask"] if s["mask"] is not None else torch.ones(n, n, dtype=torch.bool, device="cuda").tril()
                sc[:, c:].masked_fill_(~see, -math.inf)
                att[part, h] = sc.softmax(-1) @ vv
        x = x + att.reshape(-1, d) @ W["wo"].t()
        g, u = (_norm(x, W["ffn_norm"], cfg["rms_eps"]) @ W["w_gate_up"].t()).chunk(2, -1)
        x = x + (torch.nn.functional.silu(g) * u) @ W["w_down"].t()
    return _norm(x, w["final_norm"].double(), cfg["rms_eps"])


def _draft_scores(w, cfg, root, h):
    """Scores of the beam search over the drafter, 64 bits, one sequence at a time."""
    out = []
    uw = torch.cat([w["rnn_u"], w["rnn_w"]], 1).double()
    head = [(w[f"head_w.{l}"].double(), w[f"head_b.{l}"].double()) for l in range(cfg["n_head_layers"])]
    proj = w["draft_out"].double()
    for b in range(len(root)):
        s, score = w["tok_emb"][root[b]].double()[None], torch.zeros(1, dtype=torch.float64, device="cuda")
        for call in range(cfg["beam_length"]):
            x = torch.cat([s, h[b].double().expand(len(s), -1)], 1)
            for A, c in head:
                x = x + torch.nn.functional.silu(x @ A.t() + c)
            total = (score[:, None] + (x @ proj.t()).log_softmax(-1)).reshape(-1)
            score, at = total.topk(cfg["beam_width"])
            e = w["tok_emb"][at % cfg["vocab"]].double()
            s = torch.nn.functional.silu(torch.cat([s[at // cfg["vocab"]], e], 1) @ uw.t() + w["rnn_b"].double())
        out.append(score)
    return torch.stack(out)


def _tree(root, beams):
    """Packed rows of one sequence's candidates: tokens, depths and the ancestor mask."""
    tokens, depth, above, at = [int(root)], [0], [[0]], {}
    for r in beams.tolist():
        up = above[0]
        for j in range(len(r)):
            key = tuple(r[:j + 1])
            if key not in at:
                at[key] = len(tokens)
                tokens.append(r[j])
                depth.append(j + 1)
                above.append(up + [at[key]])
            up = above[at[key]]
    return tokens, depth, above


def exact(case, seed):
    p = _plan(case, seed)
    cfg, B, V, d = p["cfg"], case["batch"], p["cfg"]["vocab"], p["cfg"]["d_model"]
    w = _weights(cfg, p["succ"], seed)
    lm = w["lm_head"].double()
    H, hd, room = cfg["n_heads"], d // cfg["n_heads"], cfg["max_ctx"]
    dev = lambda v: torch.as_tensor(np.asarray(v, dtype=np.int64)).cuda()
    if case["kind"] == "prompt":
        seqs = [dict(tokens=dev(t), pos=torch.arange(len(t), device="cuda"), mask=None, ctx=0) for t in p["prompts"]]
        kv = torch.zeros(cfg["n_layers"], 2, B, H, room, hd, dtype=torch.float64, device="cuda")
        x = _forward(w, cfg, seqs, keep=kv)
        x = x[dev(np.cumsum([len(t) for t in p["prompts"]]) - 1)]
        return dict(ctx=None, root=None, hidden=x, logits=x @ lm.t(), kv=kv)
    dt = torch.float32 if cfg["dtype"] == "fp32" else torch.bfloat16
    cache = _cache_fill(torch.empty(cfg["n_layers"], 2, B, H, room, hd, dtype=dt, device="cuda"), cfg, seed)
    seqs, last = [], []
    for b in range(B):
        c, t, path = int(p["ctx"][b]), int(p["root"][b]), []
        if case["kind"] == "ar":
            for _ in range(case["steps"]):
                path.append(t)
                t = int(p["succ"][t])
            tokens, depth, above = [], [], []
            last.append(len(path) - 1)
        else:
            for s in p["steps"][:-1]:
                for _ in range(1 + s["took"][b]):
                    path.append(t)
                    t = int(p["succ"][t])
            tokens, depth, above = _tree(t, p["steps"][-1]["beams"][b])
            end = 0                                  # the node that acceptance ends at
            for _ in range(p["steps"][-1]["took"][b]):
                t = int(p["succ"][t])
                end = next(i for i in range(len(tokens)) if tokens[i] == t and len(above[i]) > 1 and above[i][-2] == end)
            last.append(len(path) + end)
        n = len(path)
        mask = np.zeros((n + len(tokens), n + len(tokens)), dtype=bool)
        mask[:n, :n] = np.tril(np.ones((n, n), dtype=bool))
        mask[n:, :n] = True
        for i, up in enumerate(above):
            mask[n + i, [n + j for j in up]] = True
        seqs.append(dict(tokens=dev(path + tokens), pos=dev(list(range(c, c + n)) + [c + n + j for j in depth]), ctx=c,
                         mask=torch.from_numpy(mask).cuda(), skip=n))
    x = _forward(w, cfg, seqs, cache)
    parts = x.split([len(s["tokens"]) for s in seqs])
    h = torch.stack([q[i] for q, i in zip(parts, last)])
    if case["kind"] == "ar":
        return dict(tokens=[None] * case["steps"], ctx=None, root=None, hidden=h, logits=h @ lm.t())
    rows = [q[s["skip"]:] for q, s in zip(parts, seqs)]
    if case["kind"] == "step":
        return dict(accepted=[[None] * 3 for _ in p["steps"]], ctx=None, root=None, hidden=h, logits=torch.cat(rows) @ lm.t())
    nmax = 1 + case["beam_width"] * case["beam_length"]
    hidden = torch.zeros(B, nmax, d, dtype=torch.float64, device="cuda")
    logits = torch.zeros(B, nmax, V, dtype=torch.float64, device="cuda")
    for b, q in enumerate(rows):
        hidden[b, :len(q)] = q
        logits[b, :len(q)] = q @ lm.t()
    scores = _draft_scores(w, cfg, p["root"].tolist(), _hidden(cfg, B, seed))
    return dict(drafted=None, scores=scores, packed=[None] * 6, argmax=None, rows=hidden, logits=logits, accepted=[None] * 3,
                ctx=None, root=None, hidden=h)
