"""The calls a program built on this library makes, as measurable cases.

A case is one call (or one chain of calls) through the public entry points on a model of one of
the repository's shapes: the layer search after a verification, the verification pass, a draft
token through the layer-skipped model, the prompt prefill, a round of non-greedy decoding, and
the whole greedy loop on the small models.

Models are random-init with three properties of trained checkpoints that plain random weights
lack, so that the outputs are well defined: the layers differ in importance (the output
projections of M "weak" layers are scaled down, as the redundant layers of a trained model are,
so a search has a set to find and is not decided by rounding), the embedding is a sizeable part
of the residual stream, and the LM head prefers one successor per token (a bigram table mixed
into it), so that greedy tokens are not near-ties and drafts are accepted at a realistic rate.
"""
import dataclasses
import math
import random

import torch

import datagen
import paper_2505_24196_b200 as clasp

WEAK = 0.1          # scale of a weak layer's contribution to the residual stream
BIGRAM = 14.0       # logit of a token's preferred successor (the rest are about N(0, 1.3))
TEMPERATURE = 1.0
MAX_ROWS = 128      # rows per call the repository's own benchmark and sweeps configure


def _case(name, kind, model, **kw):
    c = {"name": name, "kind": kind, "model": model, "layers": 0, "ctx": 0, "M": 0, "T": 1, "rows": 0, "chunk": MAX_ROWS,
         "K": 4, "new": 0}
    c.update(kw)
    return c


def listed():
    return [
        # the small fp32 model (BASELINE config: 64-token context, M = 2): latency of one search
        _case("tiny-search", "search", "tiny", ctx=64, M=2),
        # the same model's whole loop: 64-token prompt, 32 new tokens, draft length 4, search every round
        _case("tiny-generate", "generate", "tiny", ctx=64, M=2, new=32),
        # the small bf16 model of the tests, the bench's quick workload with an odd context
        _case("mini8b-search", "search", "mini8b", ctx=117, M=2),
        # the headline: one search per verification on the 8B shape
        _case("8b-search-c512", "search", "8b", ctx=512, M=12),
        # several objective positions: M x T candidate rows through every layer
        _case("8b-search-c2048-t4", "search", "8b", ctx=2048, M=12, T=4),
        # the far end of the context sweep
        _case("8b-search-c8192-t8", "search", "8b", ctx=8192, M=12, T=8),
        # the 70B layer shape (16 of its 80 layers) with as many candidate rows as its M = 32 search carries
        _case("70b-layers-search", "search", "70b", layers=16, ctx=1024, M=8, T=4),
        # one draft token through the 20 kept layers and the head
        _case("8b-draft", "draft", "8b", ctx=530, M=12),
        # verification of four drafts and the pending token
        _case("8b-verify", "verify", "8b", ctx=530, rows=5),
        # a prompt fed in the benchmark's chunks of 128 rows
        _case("8b-prefill-512-by-128", "prefill", "8b", rows=512, chunk=128),
        # a long, ragged prompt fed in one call by a context configured for it
        _case("8b-prefill-1999", "prefill", "8b", rows=1999, chunk=2048),
        # one round of non-greedy decoding: K sampled drafts, their verification, accept / resample
        _case("8b-sample-round", "sample", "8b", ctx=700, M=12, K=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "verify", "draft", "prefill", "prefill", "sample", "generate"])
    if kind == "generate":
        c = _case("", kind, rng.choice(["tiny", "small", "mini8b"]), ctx=_log_int(rng, 16, 160), K=rng.randint(2, 8),
                  new=rng.randint(8, 40))
        c["M"] = rng.randint(1, datagen.CONFIGS[c["model"]].L // 2)
    elif kind == "prefill":
        n = _log_int(rng, 24, 1990)
        c = _case("", kind, rng.choice(["mini8b", "8b", "8b"]), rows=n, chunk=rng.choice([128, 256, 512, 2048]))
        if n > 700 and c["chunk"] < 256:
            c["chunk"] = 256
    else:
        model = rng.choice(["tiny", "small", "mini8b", "8b", "8b", "8b", "70b"])
        cfg = datagen.CONFIGS[model]
        layers = rng.randint(4, 14) if model == "70b" else 0
        n_layers = layers or cfg.L
        top = 160 if cfg.dtype == "fp32" else 8000 if kind == "search" else 3000
        c = _case("", kind, model, layers=layers, ctx=_log_int(rng, 24, top))
        c["M"] = rng.randint(1, max(1, n_layers // 2))
        if kind == "search":
            c["T"] = rng.choice([1, 1, 1, 2, 3, 4, 5, 6, 7, 8])
            c["T"] = max(1, min(c["T"], MAX_ROWS // c["M"]))
        elif kind == "verify":
            c["rows"] = rng.randint(2, 9)
        elif kind == "sample":
            c["K"] = rng.randint(1, 7)
    del c["name"]
    return c


def _shape(case):
    cfg = datagen.CONFIGS[case["model"]]
    return dataclasses.replace(cfg, L=case["layers"]) if case["layers"] else cfg


def _weights(cfg, seed, weak, dev):
    """Layers and head of a random model of this shape, on the device."""
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    dt = cfg.torch_dtype

    def normal(shape, std):
        return torch.empty(shape, dtype=dt, device=dev).normal_(0.0, std, generator=g)

    d, f = cfg.d_model, cfg.d_ffn
    # projections of unit-variance rows to a standard deviation of 1.28 whatever the width (0.02 at 4096 columns)
    std_in = 1.28 / math.sqrt(d)
    layers = []
    for l in range(cfg.L):
        s = (WEAK if l in weak else 1.0) / math.sqrt(2.0 * cfg.L)
        layers.append({
            "attn_norm": 1.0 + 0.1 * torch.randn(d, device=dev, generator=g),
            "wq": normal((cfg.q_dim, d), std_in), "wk": normal((cfg.kv_dim, d), std_in),
            "wv": normal((cfg.kv_dim, d), std_in), "wo": normal((d, cfg.q_dim), s * 1.28 / math.sqrt(cfg.q_dim)),
            "mlp_norm": 1.0 + 0.1 * torch.randn(d, device=dev, generator=g),
            "w_gate": normal((f, d), std_in), "w_up": normal((f, d), std_in), "w_down": normal((d, f), s * 1.28 / math.sqrt(f))})
    head = {"embed": normal((cfg.vocab, d), 1.0), "final_norm": 1.0 + 0.1 * torch.randn(d, device=dev, generator=g),
            "lm_head": normal((cfg.vocab, d), std_in)}
    successor = torch.randperm(cfg.vocab, device=dev, generator=g)
    head["lm_head"].index_add_(0, successor, head["embed"], alpha=BIGRAM / (0.7 * d))
    return layers, head, g


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    cfg, kind, C0, M, T, K = _shape(case), case["kind"], case["ctx"], case["M"], case["T"], case["K"]
    weak = set(random.Random(seed).sample(range(cfg.L), M))
    layers, head, g = _weights(cfg, seed, weak, dev)
    max_ctx = {"prefill": case["rows"], "generate": C0 + case["new"] + 2 * (K + 1)}.get(kind, C0 + 16)
    max_rows = case["chunk"] if kind == "prefill" else MAX_ROWS
    ccfg = clasp.make_config(cfg, max_ctx=max_ctx, max_rows=max_rows, max_M=max(M, 1), max_T=T, max_head_rows=16)
    eng = clasp.Clasp(ccfg, device=dev)
    eng.load_layers(0, layers)
    eng.load_head(head)
    kv = clasp.KVCache(ccfg, device=dev)
    st = {"case": case, "cfg": cfg, "eng": eng, "kv": kv, "layers": layers, "head": head}
    if kind not in ("prefill", "generate"):
        # a verified context: keys and values as the projections of unit-variance rows give them
        kv.k.normal_(0.0, 1.28, generator=g)
        kv.v.normal_(0.0, 1.28, generator=g)
    n_tok = {"search": T, "prefill": case["rows"], "generate": C0, "verify": case["rows"]}.get(kind, 1)
    tokens = torch.randint(0, cfg.vocab, (n_tok,), device=dev, dtype=torch.int32, generator=g)
    mask = bytes(1 if l in weak else 0 for l in range(cfg.L))

    def successors(first, n):
        """The greedy continuation of `first` under the full model, as drafts for a verification."""
        toks = torch.empty(n + 1, dtype=torch.int32, device=dev)
        toks[:1] = first
        for k in range(n):
            eng.draft_forward(bytes(cfg.L), toks[k:k + 1], C0 + k, kv, toks[k + 1:k + 2])
        return toks

    if kind == "search":
        _, hid = eng.verify(tokens, C0, kv, 1)          # [T, L+1, d]: the objective's hidden states
        st["hidden"], st["objective"] = hid, tokens
    elif kind == "verify":
        n = case["rows"]
        st["tokens"] = successors(tokens[:1], n - 1)
        st["hidden"] = torch.empty((n, cfg.L + 1, cfg.d_model), dtype=torch.float32, device=dev)
        st["argmax"] = torch.empty(n, dtype=torch.int32, device=dev)
    elif kind == "prefill":
        st["tokens"] = tokens
        last = (case["rows"] - 1) % case["chunk"] + 1
        st["hidden"] = torch.empty((last, cfg.L + 1, cfg.d_model), dtype=torch.float32, device=dev)
        st["argmax"] = torch.empty(1, dtype=torch.int32, device=dev)
    elif kind == "draft":
        st["tokens"], st["mask"] = tokens, mask
        st["out"] = torch.empty(1, dtype=torch.int32, device=dev)
        st["prob"] = torch.empty(1, dtype=torch.float32, device=dev)
    elif kind == "sample":
        V = cfg.vocab
        st["tokens"] = torch.cat([tokens, tokens.new_zeros(K)])
        st["mask"] = mask
        st["q"] = torch.empty((K, V), dtype=torch.float32, device=dev)
        st["p"] = torch.empty((K + 1, V), dtype=torch.float32, device=dev)
        st["n_acc"] = torch.zeros(1, dtype=torch.int32, device=dev)
        st["committed"] = torch.zeros(K + 1, dtype=torch.int32, device=dev)
        st["hidden"] = torch.empty((K + 1, cfg.L + 1, cfg.d_model), dtype=torch.float32, device=dev)
        st["seed"] = seed
    elif kind == "generate":
        st["tokens"] = tokens.tolist()
        st["dec"] = clasp.SelfSpeculativeDecoder(eng, kv, M=M, K=K)
    return st


def run(st):
    case, cfg, eng, kv = st["case"], st["cfg"], st["eng"], st["kv"]
    kind, C0 = case["kind"], case["ctx"]
    if kind == "search":
        d = cfg.d_model
        return eng.dp_search(st["hidden"], d, (cfg.L + 1) * d, kv, C0, C0, case["T"], case["M"])
    if kind == "verify":
        n = case["rows"]
        eng.verify(st["tokens"], C0, kv, n, hidden_out=st["hidden"], argmax_out=st["argmax"])
        return {"argmax": st["argmax"], "hidden": st["hidden"], "k": kv.k[:, C0:C0 + n], "v": kv.v[:, C0:C0 + n]}
    if kind == "prefill":
        n, step = case["rows"], case["chunk"]
        for s in range(0, n, step):
            last = s + step >= n
            eng.verify(st["tokens"][s:s + step], s, kv, 1 if last else 0, want_hidden=last,
                       hidden_out=st["hidden"] if last else None, argmax_out=st["argmax"])
        return {"argmax": st["argmax"], "hidden": st["hidden"], "k": kv.k, "v": kv.v}
    if kind == "draft":
        eng.draft_forward(st["mask"], st["tokens"], C0, kv, st["out"], st["prob"])
        return {"token": st["out"], "prob": st["prob"], "k": kv.k[:, C0:C0 + 1], "v": kv.v[:, C0:C0 + 1]}
    if kind == "sample":
        K, tok = case["K"], st["tokens"]
        for k in range(K):
            eng.draft_sample(st["mask"], tok[k:k + 1], C0 + k, kv, TEMPERATURE, st["seed"], 1, tok[k + 1:k + 2], st["q"][k])
        eng.verify_sample(tok, C0, kv, K, st["q"], TEMPERATURE, st["seed"], 1, st["p"], st["n_acc"], st["committed"],
                          st["hidden"])
        return {"drafts": tok, "q": st["q"], "p": st["p"], "n_acc": st["n_acc"], "committed": st["committed"],
                "hidden": st["hidden"], "k": kv.k[:, C0:C0 + K + 1], "v": kv.v[:, C0:C0 + K + 1]}
    dec = st["dec"]
    toks = dec.generate(st["tokens"], case["new"])
    return {"tokens": torch.tensor(toks), "hidden": dec.hidden, "S": torch.tensor(list(dec.mask_host)),
            "k": kv.k[:, :C0], "v": kv.v[:, :C0]}


def _layer_pass(cfg, rows, keys):
    """Bytes and operations of one layer over `rows` rows that see `keys` positions in all on average."""
    esz = 4 if cfg.dtype == "fp32" else 2
    mats = cfg.layer_matrix_bytes()
    return (mats + 2 * keys * cfg.kv_dim * esz + 8 * rows * cfg.d_model,
            2 * rows * mats // esz + 4 * rows * keys * cfg.q_dim)


def work(case):
    cfg, kind, C0, M, T, K = _shape(case), case["kind"], case["ctx"], case["M"], case["T"], case["K"]
    esz = 4 if cfg.dtype == "fp32" else 2
    head = (cfg.vocab * cfg.d_model * esz, 2 * cfg.vocab * cfg.d_model)
    b = f = 0

    def forward(n_layers, rows, keys, head_rows):
        nonlocal b, f
        lb, lf = _layer_pass(cfg, rows, keys)
        b += n_layers * (lb + 2 * rows * cfg.kv_dim * esz)
        f += n_layers * lf
        if head_rows:
            b += head[0]
            f += head[1] * head_rows

    def search():
        nonlocal b, f
        for i in range(2, cfg.L + 1):               # step 1 has no state to push through a layer
            n = min(i - 1, M)
            lb, lf = _layer_pass(cfg, n * T, C0 + T // 2)
            b += lb
            f += lf
        b += 4 * (cfg.L + 1) * T * cfg.d_model

    if kind == "search":
        search()
    elif kind == "verify":
        forward(cfg.L, case["rows"], C0 + case["rows"] // 2, case["rows"])
    elif kind == "draft":
        forward(cfg.L - M, 1, C0, 1)
    elif kind == "prefill":
        n, step = case["rows"], case["chunk"]
        for s in range(0, n, step):
            rows = min(step, n - s)
            forward(cfg.L, rows, s + rows // 2, 1 if s + step >= n else 0)
        b += 4 * ((n - 1) % step + 1) * (cfg.L + 1) * cfg.d_model
    elif kind == "sample":
        for k in range(K):
            forward(cfg.L - M, 1, C0 + k, 1)
        forward(cfg.L, K + 1, C0 + K, K + 1)
        b += 2 * (2 * K + 1) * cfg.vocab * 4
    else:
        forward(cfg.L, C0, C0 // 2, 1)
        search()
        rounds = max(1, -(-(case["new"] - 1) // (K + 1)))
        for _ in range(rounds):
            for k in range(K):
                forward(cfg.L - M, 1, C0, 1)
            forward(cfg.L, K + 1, C0, K + 1)
            search()
    return {"bytes": float(b), "flops": float(f)}


def tolerance(case):
    # relative 2-norm of whole outputs; a token or a layer of a skip set that differs is a failure.
    # fp32: the library is within 6.5e-7 (margins) and 1.8e-7 (states) of a float64 evaluation; sums of a
    # thousand products in another order differ by a few 1e-6 where margins cancel.
    # bf16: the library's two device paths (one launch per call, one launch per step), which sum in different
    # orders and round activations at different places, differ by up to 4.5e-3 (largest single value 3e-2 of the
    # root mean square) on keys and values of a forward and by 2.5e-3 on a search's states.
    if _shape(case).dtype == "fp32":
        return {"rel": 1e-5, "max": 2e-4, "differ": 0.0}
    if case["kind"] == "search":
        return {"rel": 1e-2, "max": 6e-2, "differ": 0.0}
    return {"rel": 1.8e-2, "max": 0.12, "differ": 0.0}


# ---------------------------------------------------------------- the same results in 64 bits
# Plain torch on the state's weights, cache and tokens; hidden states of an objective are computed here from its
# tokens, nothing is taken from the library but whole numbers (drafted tokens).

def _rope64(x, pos, theta):
    hd = x.shape[-1]
    inv = theta ** (-torch.arange(0, hd, 2, dtype=torch.float64, device=x.device) / hd)
    a = pos.double()[:, None, None] * inv
    lo, hi = x[..., :hd // 2], x[..., hd // 2:]
    return torch.cat([lo * a.cos() - hi * a.sin(), hi * a.cos() + lo * a.sin()], -1)


def _norm64(cfg, x, w):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + cfg.rms_eps) * w.double()


def _layer64(cfg, lw, x, pos, ck, cv, own):
    """One decoder layer over rows x [n, d] that see the keys ck, values cv and the rows `own` [n, n] says; (y, k, v)."""
    n, nq, nkv, hd = x.shape[0], cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim
    h = _norm64(cfg, x, lw["attn_norm"])
    q = _rope64((h @ lw["wq"].double().T).view(n, nq, hd), pos, cfg.rope_theta) / math.sqrt(hd)
    k = _rope64((h @ lw["wk"].double().T).view(n, nkv, hd), pos, cfg.rope_theta)
    v = (h @ lw["wv"].double().T).view(n, nkv, hd)
    ks, vs = torch.cat([ck.double(), k]), torch.cat([cv.double(), v])
    o = torch.empty_like(q)
    for g in range(nkv):
        heads = slice(g * (nq // nkv), (g + 1) * (nq // nkv))
        s = torch.einsum("nhd,cd->hnc", q[:, heads], ks[:, g])
        s[:, :, ck.shape[0]:].masked_fill_(~own, -math.inf)
        o[:, heads] = torch.einsum("hnc,cd->nhd", s.softmax(-1), vs[:, g])
    x = x + o.reshape(n, -1) @ lw["wo"].double().T
    h = _norm64(cfg, x, lw["mlp_norm"])
    act = torch.nn.functional.silu(h @ lw["w_gate"].double().T) * (h @ lw["w_up"].double().T)
    return x + act @ lw["w_down"].double().T, k, v


def _forward64(cfg, layers, head, tokens, pos0, ck, cv, skip=None, extra=None):
    """(hidden [n, L + 1, d], k, v of the rows by layer) of tokens at pos0.. over the cache; `extra`: {layer: (k, v)} after it."""
    n = tokens.numel()
    pos = torch.arange(pos0, pos0 + n, device=tokens.device)
    causal = torch.ones((n, n), dtype=torch.bool, device=tokens.device).tril()
    x = head["embed"][tokens.long()].double()
    hid, kv = [x], {}
    for l in range(cfg.L):
        if not (skip and skip[l]):
            k0, v0 = ck[l, :pos0], cv[l, :pos0]
            if extra and l in extra:
                m = extra[l][0].shape[0]
                k0 = torch.cat([k0[:pos0 - m].double(), extra[l][0]])
                v0 = torch.cat([v0[:pos0 - m].double(), extra[l][1]])
            x, k, v = _layer64(cfg, layers[l], x, pos, k0, v0, causal)
            kv[l] = (k, v)
        hid.append(x)
    return torch.stack(hid, 1), kv


def _logits64(cfg, head, x):
    h = _norm64(cfg, x, head["final_norm"])
    return torch.cat([h @ w.double().T for w in head["lm_head"].split(16384)], -1)


def _search64(cfg, layers, hid, ck, cv, C0, T, M):
    L = cfg.L
    x = hid.transpose(0, 1)                      # [L + 1, T, d]
    nan = torch.full((L + 1, M + 1), math.nan, dtype=torch.float64, device=x.device)
    D, margin = nan.clone(), nan.clone()
    D[:, 0] = 1.0

    def score(i, y):
        return torch.nn.functional.cosine_similarity(x[i], y, dim=-1, eps=1e-12).mean(-1)

    pos = torch.arange(C0, C0 + T, device=x.device)
    causal = torch.ones((T, T), dtype=torch.bool, device=x.device).tril()
    g = {0: x[0]}
    for i in range(1, L + 1):
        n = min(i - 1, M)
        new = {0: x[i]}
        if n:
            own = torch.block_diag(*[causal.double()] * n).bool()
            y, _, _ = _layer64(cfg, layers[i - 1], torch.cat([g[j] for j in range(1, n + 1)]), pos.repeat(n),
                               ck[i - 1, :C0], cv[i - 1, :C0], own)
            app = y.view(n, T, -1)
            skip = torch.stack([g[j - 1] for j in range(1, n + 1)])
            sa, ss = score(i, app), score(i, skip)
            take = sa > ss
            D[i, 1:n + 1], margin[i, 1:n + 1] = torch.where(take, sa, ss), sa - ss
            for j in range(1, n + 1):
                new[j] = app[j - 1] if take[j - 1] else skip[j - 1]
        if i <= M:
            new[i] = g[i - 1]
            D[i, i] = score(i, g[i - 1])
        g = new
    return {"S": None, "D": D, "margin": margin, "g_final": g[M]}


def exact(case, seed):
    cfg, kind, C0, M, T, K = _shape(case), case["kind"], case["ctx"], case["M"], case["T"], case["K"]
    st = prepare(case, seed)
    layers, head, kv = st["layers"], st["head"], st["kv"]
    ck, cv = kv.k.clone(), kv.v.clone()

    def stack(own):
        return tuple(torch.stack([own[l][i] for l in range(cfg.L)]) for i in (0, 1))

    if kind == "search":
        hid, _ = _forward64(cfg, layers, head, st["objective"], C0, ck, cv)
        return _search64(cfg, layers, hid, ck, cv, C0, T, M)
    if kind == "verify":
        hid, own = _forward64(cfg, layers, head, st["tokens"], C0, ck, cv)
        k, v = stack(own)
        return {"argmax": None, "hidden": hid, "k": k, "v": v}
    if kind == "prefill":
        hid, own = _forward64(cfg, layers, head, st["tokens"], 0, ck, cv)
        k, v = stack(own)
        return {"argmax": None, "hidden": hid[-st["hidden"].shape[0]:], "k": k, "v": v}
    if kind == "generate":
        tokens = torch.tensor(st["tokens"], device=ck.device)
        k, v = stack(_forward64(cfg, layers, head, tokens, 0, ck, cv)[1])
        return {"tokens": None, "hidden": None, "S": None, "k": k, "v": v}
    if kind == "draft":
        hid, own = _forward64(cfg, layers, head, st["tokens"], C0, ck, cv, skip=st["mask"])
        p = _logits64(cfg, head, hid[:, -1]).softmax(-1).max(-1).values
        for l in range(cfg.L):
            own.setdefault(l, (ck[l, C0:C0 + 1].double(), cv[l, C0:C0 + 1].double()))
        k, v = stack(own)
        return {"token": None, "prob": p, "k": k, "v": v}
    # a sampled round: the tokens are the library's draws, everything else is computed from them
    run(st)
    tokens = st["tokens"].clone()
    q, extra = [], {}
    for i in range(K):
        hid, own = _forward64(cfg, layers, head, tokens[i:i + 1], C0 + i, ck, cv, skip=st["mask"], extra=extra)
        q.append(_logits64(cfg, head, hid[:, -1]))
        extra = {l: tuple(torch.cat([extra[l][j], own[l][j]]) if l in extra else own[l][j] for j in (0, 1)) for l in own}
    hid, own = _forward64(cfg, layers, head, tokens, C0, ck, cv)
    k, v = stack(own)
    return {"drafts": None, "q": torch.cat(q), "p": _logits64(cfg, head, hid[:, -1]), "n_acc": None, "committed": None,
            "hidden": hid, "k": k, "v": v}
