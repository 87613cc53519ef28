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
from tests.util import Pair, check_search_against_oracle, kv_to_oracle, scaled_keys, search_that_applies_layer_1, tol_hidden

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
