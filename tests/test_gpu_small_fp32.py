"""The one-launch path of fp32 models that fit a cluster (csrc/small32.cuh) against one kernel per step
(CLASP_FLAG_MULTI_KERNEL, which test_gpu_parity.py and test_gpu_draft_and_loop.py compare with the oracle beside it): both
head dimensions, widths that are no multiple of a warp's stride, rows around the passes of eight, ragged key blocks, an LM
head that fits its slice and one that does not, a draft that skips every layer.  Whole calls at head dimension 128 against
the oracle; calls on either side of the limits of the path over one cache.

Both sides sum at most 704 products in fp32 in different orders: the expected difference is about sqrt(704) * 6e-8 = 2e-6
of a value's scale, growing over the layers; 2e-5 leaves a factor of ten."""
import dataclasses

import numpy as np
import pytest
import torch

import datagen
import paper_2505_24196_b200 as clasp
from oracle import clasp_oracle as orc
from tests.util import Pair, check_search_against_oracle, close_hidden, rel_l2, tol_hidden

pytestmark = pytest.mark.gpu
TOL = 2e-5
TINY = datagen.CONFIGS["tiny"]
MODELS = {
    "hd64": TINY,
    "hd128": dataclasses.replace(TINY, name="hd128", L=5, d_model=192, n_q_heads=2, n_kv_heads=1, head_dim=128, d_ffn=520,
                                 vocab=1000),
    "big-head": dataclasses.replace(TINY, name="big-head", L=3, d_ffn=704, vocab=3000),
}


class Two:
    """The same weights in a context of either path."""

    def __init__(self, cfg, max_ctx=200, max_rows=64):
        self.cfg = cfg
        layers = [{k: v.cuda().contiguous() for k, v in datagen.layer_weights(cfg, l, "cpu").items()} for l in range(cfg.L)]
        head = {k: v.cuda().contiguous() for k, v in datagen.head_weights(cfg, "cpu").items()}
        self.layers, self.head = layers, head
        self.eng = []
        for flags in (0, clasp.FLAG_MULTI_KERNEL):
            e = clasp.Clasp(clasp.make_config(cfg, max_ctx=max_ctx, max_rows=max_rows, max_M=cfg.L, max_T=8, max_head_rows=16,
                                             flags=flags))
            e.load_layers(0, layers)
            e.load_head(head)
            self.eng.append(e)

    def caches(self, ctx):
        out = []
        for e in self.eng:
            kv = clasp.KVCache(e.cfg)
            kv.k[:, :ctx] = datagen.normal_rows(91, 0, tuple(kv.k[:, :ctx].shape)).cuda()
            kv.v[:, :ctx] = datagen.normal_rows(91, 1, tuple(kv.v[:, :ctx].shape)).cuda()
            out.append(kv)
        return out


@pytest.fixture(scope="module", params=list(MODELS))
def two(request):
    return Two(MODELS[request.param])


def close(a, b):
    return rel_l2(a.double().cpu().numpy(), b.double().cpu().numpy()) < TOL


@pytest.mark.parametrize("n,ctx", [(1, 0), (1, 31), (2, 32), (3, 7), (8, 120), (9, 0), (33, 100), (64, 64)])
def test_forward(two, n, ctx):
    toks = datagen.token_ids(two.cfg, n).to(torch.int32).cuda()
    heads = min(n, 9)
    res = []
    for e, kv in zip(two.eng, two.caches(ctx)):
        n0 = e.launch_count()
        am, hid = e.verify(toks, ctx, kv, heads)
        res.append((am.cpu(), hid, kv, e.launch_count() - n0))
        assert e.device_status() == 0
    (am1, h1, kv1, n1), (am2, h2, kv2, n2) = res
    assert n1 <= 4 < n2                       # one launch (and three when the head does not fit)
    assert close(h1, h2) and close(kv1.k, kv2.k) and close(kv1.v, kv2.v)
    assert torch.equal(am1, am2)


@pytest.mark.parametrize("skip", ["none", "some", "all"])
def test_draft(two, skip):
    L = two.cfg.L
    mask = {"none": bytes(L), "some": bytes(l % 2 for l in range(L)), "all": bytes([1] * L)}[skip]
    res = []
    for e, kv in zip(two.eng, two.caches(50)):
        tok = torch.tensor([5], dtype=torch.int32, device="cuda")
        out, prob = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(1, device="cuda")
        e.draft_forward(mask, tok, 50, kv, out, prob)
        assert e.device_status() == 0
        res.append((int(out), float(prob), kv))
    assert res[0][0] == res[1][0] and abs(res[0][1] - res[1][1]) < 1e-5 * res[1][1]
    assert close(res[0][2].k, res[1][2].k) and close(res[0][2].v, res[1][2].v)


@pytest.mark.parametrize("M,T,ctx", [(1, 1, 0), (2, 1, 63), (3, 1, 64), (2, 3, 33), (3, 8, 150)])
def test_search(two, M, T, ctx):
    cfg = two.cfg
    hid = datagen.normal_rows(92, M * 10 + T, (T, cfg.L + 1, cfg.d_model)).to(torch.float32).cuda()
    res = []
    for e, kv in zip(two.eng, two.caches(ctx)):
        res.append(e.dp_search(hid, cfg.d_model, (cfg.L + 1) * cfg.d_model, kv, ctx, ctx, T, M))
        assert e.device_status() == 0
    a, b = res
    # margins of random states are of the order of 1 / sqrt(d): far from ties
    assert torch.equal(a["S"], b["S"]) and close(a["g_final"], b["g_final"])
    for key in ("D", "margin"):
        x, y = a[key], b[key]
        assert torch.equal(torch.isnan(x), torch.isnan(y))
        ok = ~torch.isnan(y)
        assert float((x[ok] - y[ok]).abs().max() if ok.any() else 0.0) < TOL


@pytest.mark.parametrize("M,T,ctx", [(1, 1, 40), (2, 3, 64), (3, 2, 33), (3, 8, 150)])
def test_pruned_search_is_the_same_bits(two, M, T, ctx):
    """CLASP_FLAG_PRUNE: skip set, g[L][M] and every cell that can reach (L, M) unchanged, the others NaN; M = L too
    (no state is ever pushed through a layer).  A context with the flag keeps the one-launch path for everything."""
    cfg = two.cfg
    L = cfg.L
    hid = datagen.normal_rows(93, M * 10 + T, (T, L + 1, cfg.d_model)).to(torch.float32).cuda()
    e, kv = two.eng[0], two.caches(ctx)[0]
    p = clasp.Clasp(clasp.make_config(cfg, max_ctx=200, max_rows=64, max_M=L, max_T=8, max_head_rows=16, flags=clasp.FLAG_PRUNE))
    p.load_layers(0, two.layers)
    p.load_head(two.head)
    try:
        for m in (M, L):
            n0 = p.launch_count()
            a, b = (x.dp_search(hid, cfg.d_model, (L + 1) * cfg.d_model, kv, ctx, ctx, T, m) for x in (e, p))
            assert p.launch_count() - n0 == 1
            assert p.device_status() == 0 and e.device_status() == 0
            i, j = torch.meshgrid(torch.arange(L + 1, device="cuda"), torch.arange(m + 1, device="cuda"), indexing="ij")
            out = (j < m - (L - i)) & (j > 0)
            assert torch.equal(a["S"], b["S"]) and torch.equal(a["g_final"], b["g_final"])
            for key in ("D", "margin"):
                want = a[key].masked_fill(out, float("nan"))
                assert torch.equal(torch.isnan(b[key]), torch.isnan(want)), (m, key)
                assert torch.equal(b[key].nan_to_num(7.0), want.nan_to_num(7.0)), (m, key)
        n0 = p.launch_count()
        p.verify(torch.zeros(4, dtype=torch.int32, device="cuda"), ctx, kv, 1)
        assert p.launch_count() - n0 <= 4
    finally:
        p.close()


def test_cosines_keep_small_columns():
    """Eq. 2's sums over many columns: 128 columns of 1 and 1408 of about 2^-12.5, of the other sign in one state.  An
    addend of four small products is below half an ulp of a lane's fp32 sum, all of them together move the cosine by
    6.4e-7; partial sums of at most four products leave 2^-24 or so."""
    cfg = dataclasses.replace(TINY, name="wide-row", L=2, d_model=1536, n_q_heads=1, n_kv_heads=1, head_dim=64, d_ffn=32, vocab=64)
    e = clasp.Clasp(clasp.make_config(cfg, max_ctx=8, max_rows=4, max_M=2, max_T=1))
    e.load_layers(0, [{k: v.cuda().contiguous() for k, v in datagen.layer_weights(cfg, l, "cpu").items()} for l in range(cfg.L)])
    small = torch.tensor(1.7e-4)
    x0 = torch.ones(1536)
    x0[128:] = small
    x1 = x0.clone()
    x1[128:] = -small
    hid = torch.stack([x0, x1, x0]).cuda()
    n0 = e.launch_count()
    r = e.dp_search(hid, 1536, 0, clasp.KVCache(e.cfg), 0, 0, 1, 2)
    assert e.launch_count() - n0 == 1 and e.device_status() == 0
    a, b = x1.double(), x0.double()
    want = float(a @ b / (a.norm() * b.norm()))
    assert abs(float(r["D"][1, 1]) - want) < 2.0 ** -22
    e.close()


def test_norm_keeps_small_columns():
    """The same for the sum of squares of an RMSNorm: 128 columns of 1 and 1408 of 2^-12.5 are 6.2e-7 of the sum, half that
    of the scale.  wv of one column copies the normed column 0 into the value cache."""
    cfg = dataclasses.replace(TINY, name="wide-row", L=1, d_model=1536, n_q_heads=1, n_kv_heads=1, head_dim=64, d_ffn=32, vocab=64)
    lw = {k: v.cuda().contiguous() for k, v in datagen.layer_weights(cfg, 0, "cpu").items()}
    head = {k: v.cuda().contiguous() for k, v in datagen.head_weights(cfg, "cpu").items()}
    lw["attn_norm"].fill_(1.0)
    lw["wv"].zero_()
    lw["wv"][:, 0] = 1.0
    head["embed"][:, :128] = 1.0
    head["embed"][:, 128:] = 1.7e-4
    e = clasp.Clasp(clasp.make_config(cfg, max_ctx=8, max_rows=4, max_M=1, max_T=1))
    e.load_layers(0, [lw])
    e.load_head(head)
    kv = clasp.KVCache(e.cfg)
    n0 = e.launch_count()
    e.verify(torch.zeros(1, dtype=torch.int32, device="cuda"), 0, kv, 0)
    assert e.launch_count() - n0 == 1 and e.device_status() == 0
    row = head["embed"][0].double()
    want = float(torch.rsqrt((row * row).mean() + cfg.rms_eps))
    assert abs(float(kv.v[0, 0, 0, 0]) / want - 1.0) < 2.0 ** -23
    e.close()


@pytest.mark.parametrize("flags", [0, clasp.FLAG_MULTI_KERNEL], ids=["one-launch", "per-step"])
def test_head_dimension_128_against_the_oracle(flags):
    """Verification, draft and search of an fp32 model with head dimension 128 (tolerances of test_gpu_parity.py)."""
    cfg = MODELS["hd128"]
    p = Pair(cfg, max_ctx=96, max_rows=64, max_M=3, max_T=2, max_head_rows=4, flags=flags)
    n, L, d, M, T = 41, cfg.L, cfg.d_model, 3, 2
    toks = datagen.token_ids(cfg, n)
    oc, kv = p.new_oracle_cache(), p.new_kv()
    am_o, hid_o, logits = orc.verify_forward(p.oracle, toks.numpy(), oc, 0)
    am, hid = p.engine.verify(toks.cuda(), 0, kv, 4)
    assert close_hidden(hid.cpu().numpy(), hid_o, tol_hidden(cfg))
    top = np.sort(logits[-4:], axis=-1)
    assert (am.cpu().numpy() == am_o[-4:])[top[:, -1] - top[:, -2] > 1e-3 * np.abs(logits).max()].all()
    p0 = n - T
    ref = orc.dp_search(p.oracle, np.transpose(hid_o[p0:n], (1, 0, 2)), oc, p0, p0, M)
    res = p.engine.dp_search(hid[p0], d, (L + 1) * d, kv, p0, p0, T, M)
    D, margin, S = (res[k].cpu().numpy() for k in ("D", "margin", "S"))
    assert np.array_equal(np.isnan(D), np.isnan(ref["D"]))
    check_search_against_oracle(D, margin, S, res["g_final"].cpu().numpy(), ref, L, M, tol_hidden(cfg))
    forced = torch.from_numpy(ref["choice"].copy()).cuda()
    rf = p.engine.dp_search(hid[p0], d, (L + 1) * d, kv, p0, p0, T, M, forced_choice=forced)
    ok = ~np.isnan(ref["D"])
    np.testing.assert_allclose(rf["D"].cpu().numpy()[ok], ref["D"][ok], atol=1e-6)
    assert close_hidden(rf["g_final"].cpu().numpy(), ref["g"][L, M], tol_hidden(cfg))
    assert p.engine.device_status() == 0
    p.engine.close()


def test_one_cache_on_both_sides_of_the_limits():
    """A prompt in pieces of 128, 129 and 51 rows, then verifications and single rows around the limits: 128 rows, 2048
    positions, 65536 scores (rows x heads x keys).  The launches of a call tell its route; every piece continues the cache of
    the one before, whichever route wrote it."""
    cfg = dataclasses.replace(TINY, L=2)
    two = Two(cfg, max_ctx=2100, max_rows=129)
    caches = two.caches(0)
    toks = datagen.token_ids(cfg, 2100).to(torch.int32).cuda()
    pos, routes = 0, []
    for n in [128, 129, 51] + [129] * 13 + [9, 8, 45, 1, 1, 7]:
        keys = pos + n
        one = n <= 128 and keys <= 2048 and n * cfg.n_q_heads * keys <= 65536
        res = []
        for e, kv in zip(two.eng, caches):
            n0 = e.launch_count()
            am, hid = e.verify(toks[pos:keys], pos, kv, 1)
            res.append((am, hid, e.launch_count() - n0))
            assert e.device_status() == 0
        assert (res[0][2] == 1) == one and res[1][2] > 10, (n, keys, res[0][2])
        assert close(res[0][1], res[1][1]) and torch.equal(res[0][0], res[1][0]), (n, keys)
        routes.append(one)
        pos = keys
    assert routes == [True, False, True] + [False] * 13 + [False, True, False, True, False, False]
    assert close(caches[0].k[:, :pos], caches[1].k[:, :pos]) and close(caches[0].v[:, :pos], caches[1].v[:, :pos])
