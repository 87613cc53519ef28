"""Epilogues, Eq. 2 step and attention of the persistent kernel where the split of their work changes with the rows and the
shape: one to four and more passes of the workers over a CTA's rows (32, 64 or 128 rows a pass for slices of 8 to 64
features), rows that fill a pass or leave one over, pair blocks of 128 (row, query head) pairs whose own keys start inside a
state, one and several key runs per CTA.  Against the oracle, row by row: a bf16 operand is off by 2^-9 / sqrt(3) (rms) and a
branch of the layer has two or three of them in a row, so rows are within about 3e-3; 6e-3 is allowed."""
import dataclasses

import numpy as np
import pytest
import torch

import datagen
import paper_2505_24196_b200 as clasp
from oracle import clasp_oracle as orc
from tests.util import (Pair, check_search_against_oracle, kv_to_oracle, rel_l2, scaled_keys, search_that_applies_layer_1,
                        tol_hidden)

pytestmark = pytest.mark.gpu
MINI = datagen.CONFIGS["mini8b"]
MODELS = {
    "slices-of-8": MINI,                                          # four query heads per kv head
    "hd64": datagen.CONFIGS["small"],
    # slices of 56 and 64 features, eight query heads per kv head
    "slices-of-64": dataclasses.replace(MINI, name="wide-slice", d_model=8192, n_q_heads=16, n_kv_heads=2, d_ffn=512, vocab=64, L=2),
}
MAX_CTX = 900


@pytest.fixture(scope="module", params=list(MODELS))
def pair(request):
    p = Pair(MODELS[request.param], max_ctx=MAX_CTX, max_rows=128, max_M=3 if request.param != "slices-of-64" else 2, max_T=43,
             gen_device="cuda")
    yield p
    assert p.engine.device_status() == 0
    p.engine.close()


@pytest.mark.parametrize("S,T,C", [
    (1, 128, 0),       # a prompt of one call: every pair block sees own keys only
    (1, 33, 520),      # one row past a pass of 32
    (25, 5, 40),       # states that straddle the pair blocks
    (9, 14, 770),
    (128, 1, 33),
    (3, 41, 0),        # no cache: the own keys are the only chunk
])
def test_layer_rows(pair, S, T, C):
    cfg, layer = pair.cfg, 1
    kv, ocache = pair.new_kv(), pair.new_oracle_cache()
    shape = (cfg.L, MAX_CTX, cfg.n_kv_heads, cfg.head_dim)
    for t, k in ((kv.k, 0), (kv.v, 1)):
        t.copy_(datagen.normal_rows(81, k, shape).to(cfg.torch_dtype))
    kv_to_oracle(kv, MAX_CTX, ocache)
    x = datagen.normal_rows(82, S * 1000 + T, (S * T, cfg.d_model)).to(torch.float32)
    n0 = pair.engine.launch_count()
    out = pair.engine.layer_forward(layer, x.cuda(), S, T, C, C, kv, write_kv=S == 1).cpu().numpy()
    assert pair.engine.launch_count() - n0 == 2, "set-up and persistent kernel"
    xs = x.double().numpy().reshape(S, T, cfg.d_model)
    for s in sorted({0, S // 3, S // 2, S - 1}):
        ref, k_new, v_new = orc.decoder_layer(xs[s], pair.oracle.layer(layer), ocache.k[layer], ocache.v[layer], C, C, cfg)
        err = np.linalg.norm(out[s * T:(s + 1) * T] - ref, axis=1) / np.linalg.norm(ref, axis=1)
        assert err.max() < 6e-3, (s, int(err.argmax()), float(err.max()))
    if S == 1:
        for got, want in ((kv.k, k_new), (kv.v, v_new)):
            g = got[layer, C:C + T].double().cpu().numpy()
            assert np.linalg.norm(g - want) < 5e-3 * np.linalg.norm(want)


@pytest.mark.parametrize("M,T", [(1, 33), (2, 7), (3, 5), (3, 42)])
def test_search_rows(pair, M, T):
    cfg, n = pair.cfg, 64
    if M > cfg.L:
        pytest.skip("more skipped layers than the model has")
    L, d, p0 = cfg.L, cfg.d_model, n - T
    toks = datagen.token_ids(cfg, n)
    ocache, kv = pair.new_oracle_cache(), pair.new_kv()
    _, hid_o, _ = orc.verify_forward(pair.oracle, toks.numpy(), ocache, 0)
    kv.k[:, :n] = torch.from_numpy(ocache.k[:, :n]).to(cfg.torch_dtype).cuda()
    kv.v[:, :n] = torch.from_numpy(ocache.v[:, :n]).to(cfg.torch_dtype).cuda()
    x_o = np.transpose(hid_o[p0:n], (1, 0, 2))
    ref = orc.dp_search(pair.oracle, x_o, ocache, p0, p0, M)
    hid = torch.from_numpy(np.ascontiguousarray(hid_o[p0:n])).float().cuda()
    forced = torch.from_numpy(ref["choice"].copy()).cuda()
    res = pair.engine.dp_search(hid, d, (L + 1) * d, kv, p0, p0, T, M)
    D, margin, S = (res[k].cpu().numpy() for k in ("D", "margin", "S"))
    assert np.array_equal(np.isnan(D), np.isnan(ref["D"]))
    check_search_against_oracle(D, margin, S, res["g_final"].cpu().numpy(), ref, L, M, tol_hidden(cfg))
    rf = pair.engine.dp_search(hid, d, (L + 1) * d, kv, p0, p0, T, M, forced_choice=forced)
    g = rf["g_final"].cpu().numpy()
    err = np.linalg.norm(g - ref["g"][L, M], axis=1) / np.linalg.norm(ref["g"][L, M], axis=1)
    assert err.max() < tol_hidden(cfg), int(err.argmax())
    ok = ~np.isnan(ref["D"])
    np.testing.assert_allclose(rf["D"].cpu().numpy()[ok], ref["D"][ok], atol=1e-3)


@pytest.mark.parametrize("T", [1, 2, 33, 128])
def test_first_step_of_a_search(T):
    """The one cell of step 1, the mean over the objective rows of cos(x_1, x_0), against float64, and again on the same
    context (the rows' count has to be back at zero).  Sums of four fp32 products added in float64, then a handful of fp32
    operations and the mean: within 1e-6."""
    cfg = MINI
    ccfg = clasp.make_config(cfg, max_ctx=160 + T, max_rows=128, max_M=1, max_T=T)
    eng = clasp.Clasp(ccfg)
    eng.load_layers(0, [datagen.layer_weights(cfg, l, "cuda") for l in range(cfg.L)])
    kv = clasp.KVCache(ccfg)
    for seed in (1, 2, 2):
        g = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn((T, cfg.L + 1, cfg.d_model), device="cuda", generator=g).cumsum(1)
        D = eng.dp_search(x, cfg.d_model, (cfg.L + 1) * cfg.d_model, kv, 160, 160, T, 1)["D"].cpu()
        want = torch.nn.functional.cosine_similarity(x[:, 0].double(), x[:, 1].double(), dim=-1).mean()
        assert D[1, 0] == 1.0 and abs(float(D[1, 1]) - float(want)) < 1e-6
    assert eng.device_status() == 0
    eng.close()


@pytest.mark.parametrize("nq,nkv,hd,C,T", [
    (32, 32, 128, 200, 3),     # a run of the context per CTA
    (32, 32, 128, 2400, 3),    # eight or so runs per kv head: a CTA takes chunks of several heads
    (64, 64, 64, 1000, 40),
    (64, 64, 64, 2400, 3),
    (64, 16, 64, 2400, 40),    # 160 (row, query head) pairs per kv head: the form that walks consecutive chunks
    (33, 33, 128, 700, 2),     # a number of heads that does not divide the grid
])
def test_search_with_many_kv_heads(nq, nkv, hd, C, T):
    """More kv heads than leave the grid 16 chunks each: the runs of a search's attention are cut by rounds of chunks.  The search's
    best state is a layer output it computed, compared row by row with the oracle (keys scaled so that every tile counts)."""
    cfg = dataclasses.replace(MINI, name="heads", L=2, n_q_heads=nq, n_kv_heads=nkv, head_dim=hd, d_ffn=512, vocab=64)
    m = Pair(cfg, max_ctx=C, max_rows=64, max_M=1, max_T=T, gen_device="cuda")
    m.kv, m.ocache = m.new_kv(), m.new_oracle_cache()
    for t, k in ((m.kv.k, 0), (m.kv.v, 1)):
        t.copy_(datagen.normal_rows(83, k, tuple(t.shape)).to(cfg.torch_dtype))
    kv_to_oracle(m.kv, C, m.ocache)
    assert m.engine.engine_active()
    with scaled_keys(m, 0, 4):
        search_that_applies_layer_1(m, C, T, 84)
    m.engine.close()


FORWARDS = {
    "slices-of-8": MINI,
    "hd64": datagen.CONFIGS["small"],
    "slices-of-32": dataclasses.replace(datagen.CONFIGS["8b"], name="8b-l2", vocab=4096, L=2),
    # slices past 64 features: a lane quarter of the accumulator holds 32 of them instead of 16; eight query heads per kv head
    "slices-of-72": dataclasses.replace(MINI, name="wider-slice", d_model=10240, n_q_heads=16, n_kv_heads=2, d_ffn=512, vocab=2048, L=2),
}


@pytest.mark.parametrize("model", list(FORWARDS))
@pytest.mark.parametrize("n,C", [(40, 517), (64, 100)])   # (from 65 rows on the CTAs start their walks over K elsewhere)
def test_forward_rows_do_not_depend_on_the_rows_of_the_call(model, n, C):
    """The same tokens in one call, whose (row, query head) pairs need several blocks of 128, and in calls of at most one
    block: states, keys, values and logits are the same bits (verification, of 64 rows at most, and one-token decoding must
    agree)."""
    cfg, K = FORWARDS[model], 7
    per_call = 128 // (cfg.n_q_heads // cfg.n_kv_heads)
    assert n > per_call > K
    ccfg = clasp.make_config(cfg, max_ctx=MAX_CTX, max_rows=128, max_M=1, max_T=1)
    eng = clasp.Clasp(ccfg)
    eng.load_layers(0, [datagen.layer_weights(cfg, l, "cuda") for l in range(cfg.L)])
    eng.load_head(datagen.head_weights(cfg, "cuda"))
    g = torch.Generator(device="cuda").manual_seed(17)
    toks = torch.randint(0, cfg.vocab, (n,), device="cuda", dtype=torch.int32, generator=g)
    q = torch.zeros((K, cfg.vocab), device="cuda")
    k0, v0 = (torch.randn((cfg.L, C, cfg.n_kv_heads, cfg.head_dim), device="cuda", generator=g).to(torch.bfloat16) for _ in range(2))

    def call(pieces):
        kv = clasp.KVCache(ccfg)
        kv.k[:, :C], kv.v[:, :C] = k0, v0
        hidden, lo = [], 0
        for m in pieces[:-1]:
            hidden.append(eng.verify(toks[lo:lo + m].clone(), C + lo, kv, 0)[1])
            lo += m
        hidden.append(torch.empty((n - lo, cfg.L + 1, cfg.d_model), device="cuda"))
        p = torch.empty((K + 1, cfg.vocab), device="cuda")
        out = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(K + 1, dtype=torch.int32, device="cuda")
        eng.verify_sample(toks[lo:].clone(), C + lo, kv, K, q, 1.0, 5, 1, p, *out, hidden[-1])
        return {"hidden": torch.cat(hidden), "k": kv.k[:, C:C + n], "v": kv.v[:, C:C + n], "logits": p}

    whole = call([n])
    rest = n - (K + 1)
    cuts = [min(per_call, rest - lo) for lo in range(0, rest, per_call)]
    some = call(cuts + [K + 1])
    assert eng.device_status() == 0
    for key in whole:
        assert torch.equal(whole[key], some[key]), key
    eng.close()


@pytest.mark.parametrize("L", [98, 99, 101])
def test_models_of_many_layers(L):
    """The job list travels as a kernel parameter up to 99 jobs and is copied beyond: a verification has L + 1 jobs, a search
    L - 1.  Against the oracle, whose decisions the search is given."""
    cfg = dataclasses.replace(MINI, name="deep", L=L, d_model=128, n_q_heads=2, n_kv_heads=1, head_dim=64, d_ffn=128, vocab=64)
    n, T, M = 12, 2, 2
    p = Pair(cfg, max_ctx=32, max_rows=64, max_M=M, max_T=T)
    toks = datagen.token_ids(cfg, n)
    ocache, kv = p.new_oracle_cache(), p.new_kv()
    _, hid_o, _ = orc.verify_forward(p.oracle, toks.numpy(), ocache, 0)
    _, hid = p.engine.verify(toks.cuda(), 0, kv, n)
    assert p.engine.engine_active()
    assert rel_l2(hid.cpu().numpy(), hid_o) < tol_hidden(cfg)
    x_o, p0 = np.transpose(hid_o[n - T:], (1, 0, 2)), n - T
    kv.k.copy_(torch.from_numpy(ocache.k).to(cfg.torch_dtype))
    kv.v.copy_(torch.from_numpy(ocache.v).to(cfg.torch_dtype))
    ref = orc.dp_search(p.oracle, x_o, ocache, p0, p0, M)
    x = torch.from_numpy(np.ascontiguousarray(hid_o[n - T:])).float().cuda()
    res = p.engine.dp_search(x, cfg.d_model, (L + 1) * cfg.d_model, kv, p0, p0, T, M,
                             forced_choice=torch.from_numpy(ref["choice"].copy()).cuda())
    D = res["D"].cpu().numpy()
    assert np.array_equal(np.isnan(D), np.isnan(ref["D"]))
    np.testing.assert_allclose(D[~np.isnan(D)], ref["D"][~np.isnan(D)], atol=1e-3)
    assert np.array_equal(res["S"].cpu().numpy(), ref["S"])
    assert p.engine.device_status() == 0
    p.engine.close()
