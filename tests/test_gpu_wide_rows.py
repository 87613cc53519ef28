"""One decoder layer over more rows than the skinny products take (the tensor-core products and attention of
csrc/wide.cuh) against the oracle: edges of the 256-row and 256-feature tiles, ragged key tiles, several states with
their own rows only, key splits, and a row maximum that moves in mid-cache (the rescaling path).  Then the schedules of the
products (whole tiles, split tiles, both) with every row compared, and the attention by itself, with a limit that a lost low
part of an operand does not meet."""
import ctypes
import dataclasses

import numpy as np
import pytest
import torch

import datagen
import paper_2505_24196_b200 as clasp
from oracle import clasp_oracle as orc
from tests.util import Pair, close_hidden, kv_to_oracle, rel_l2, tol_hidden

pytestmark = pytest.mark.gpu
MAX_CTX, MAX_ROWS = 1300, 512


@pytest.fixture(scope="module", params=["mini8b", "small"])   # head dimension 128 and 64 (the latter: products only)
def pair(request):
    return Pair(datagen.CONFIGS[request.param], max_ctx=MAX_CTX, max_rows=MAX_ROWS, max_M=2, max_T=1)


@pytest.mark.parametrize("S,T,C,write,grow", [
    (1, 129, 0, True, False),      # one row past the skinny path, no cache
    (1, 256, 64, True, False),     # whole row tile, whole key tile
    (1, 257, 701, True, True),     # one row in the second tile; keys grow in the middle of the cache
    (26, 5, 333, False, False),    # states of a search: block-diagonal own rows, ragged pair block
    (2, 250, 1000, False, True),
])
def test_layer_over_many_rows(pair, S, T, C, write, grow):
    cfg, layer = pair.cfg, 1
    kv = pair.new_kv()
    shape = (cfg.L, MAX_CTX, cfg.n_kv_heads, cfg.head_dim)
    ck, cv = (datagen.normal_rows(61, k, shape).to(cfg.torch_dtype) for k in (0, 1))
    if grow:
        ck[:, C // 2:] *= 8        # exact in bf16 and shared by both sides: scores of the second half are 8 times larger
    kv.k.copy_(ck)
    kv.v.copy_(cv)
    ocache = pair.new_oracle_cache()
    kv_to_oracle(kv, MAX_CTX, ocache)
    x = datagen.normal_rows(62, S * 1000 + T, (S * T, cfg.d_model)).to(torch.float32)
    out = pair.engine.layer_forward(layer, x.cuda(), S, T, C, C, kv, write_kv=write).cpu().numpy()
    assert pair.engine.device_status() == 0
    xs = x.double().numpy().reshape(S, T, cfg.d_model)
    for s in {0, S // 2, S - 1}:
        ref, k_new, v_new = orc.decoder_layer(xs[s], pair.oracle.layer(layer), ocache.k[layer], ocache.v[layer], C, C, cfg)
        got = out[s * T:(s + 1) * T]
        assert close_hidden(got, ref, tol_hidden(cfg))
        # row by row: a wrong key tile or a lost rescaling moves single rows (bf16 operands leave about 3e-3)
        err = np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1)
        assert err.max() < tol_hidden(cfg), int(err.argmax())
    if write:
        assert rel_l2(kv.k[layer, C:C + T].float().cpu().numpy(), k_new) < 5e-3
        assert rel_l2(kv.v[layer, C:C + T].float().cpu().numpy(), v_new) < 5e-3
    else:
        assert torch.equal(kv.k.cpu(), ck) and torch.equal(kv.v.cpu(), cv)


def test_long_prompt_in_one_call_and_in_pieces(pair):
    """The same prompt through one wide call and through calls of 96 rows: hidden states, cache and greedy token."""
    cfg, n = pair.cfg, 450
    toks = torch.randint(0, cfg.vocab, (n,), generator=torch.Generator().manual_seed(7), dtype=torch.int32).cuda()
    kv1, kv2 = pair.new_kv(), pair.new_kv()
    am1, h1 = pair.engine.verify(toks, 0, kv1, 1)
    for s in range(0, n, 96):
        am2, h2 = pair.engine.verify(toks[s:s + 96], s, kv2, 1 if s + 96 >= n else 0)
    last = h2.shape[0]
    assert rel_l2(h1[-last:].cpu().numpy(), h2.cpu().numpy()) < tol_hidden(cfg)
    assert rel_l2(kv1.k[:, :n].float().cpu().numpy(), kv2.k[:, :n].float().cpu().numpy()) < tol_hidden(cfg)
    assert pair.engine.device_status() == 0


@pytest.mark.parametrize("n", [112, 113, 128])
def test_the_widest_calls_of_the_persistent_kernel(pair, n):
    """128 operand rows: on these narrow models a ring item's operand box would be larger than a tensor map describes."""
    cfg = pair.cfg
    toks = torch.randint(0, cfg.vocab, (n,), generator=torch.Generator().manual_seed(9), dtype=torch.int32).cuda()
    kv1, kv2 = pair.new_kv(), pair.new_kv()
    _, h1 = pair.engine.verify(toks, 0, kv1, 1)
    pair.engine.verify(toks[:64], 0, kv2, 0, want_hidden=False)
    _, h2 = pair.engine.verify(toks[64:], 64, kv2, 1)
    assert rel_l2(h1[64:].cpu().numpy(), h2.cpu().numpy()) < tol_hidden(cfg)
    assert pair.engine.device_status() == 0


def test_products_are_in_the_launch_timing(pair):
    """clasp_profile_gemm counts every tensor-core product: four per layer over many rows and the head."""
    cfg, eng = pair.cfg, pair.engine
    n, ms, nb = ctypes.c_int64(), ctypes.c_double(), ctypes.c_double()
    toks = torch.zeros(300, dtype=torch.int32, device="cuda")
    assert eng.lib.clasp_profile_gemm(eng.handle, 1, None, None, None) == 0
    eng.verify(toks, 0, pair.new_kv(), 1, want_hidden=False)
    assert eng.lib.clasp_profile_gemm(eng.handle, 0, ctypes.byref(n), ctypes.byref(ms), ctypes.byref(nb)) == 0
    assert n.value == 4 * cfg.L + 1 and ms.value > 0.0
    assert nb.value == cfg.L * cfg.layer_matrix_bytes() + cfg.vocab * cfg.d_model * 2


# deep rows (K = 8192 and more) beside few features, so that other products than the down product are split over K
DEEP = {
    "deep-qkv": dataclasses.replace(datagen.CONFIGS["8b"], name="deep-qkv", d_model=10240, n_q_heads=2, n_kv_heads=2, d_ffn=1280),
    "deep-gate": dataclasses.replace(datagen.CONFIGS["8b"], name="deep-gate", d_model=8192, n_q_heads=16, n_kv_heads=2, d_ffn=3200),
}
# (model, rows, states): what the 74 pairs of CTAs do with the 256-row tiles of q/k/v, o, gate/up and down
SCHEDULES = [
    ("mini8b", 1999, 1999),   # gate/up: 224 tiles, up to four per pair; nothing split (few chunks of K)
    ("mini8b", 1300, 26),     # gate/up: 168 tiles
    ("small", 1999, 1999),    # gate/up: 88 tiles on 74 pairs; q/k/v and o one per pair at most
    ("8b", 129, 43),          # down: all 16 tiles split, four parts each; the others whole
    ("8b", 257, 257),         # down: all 32 tiles split, two parts each
    ("8b", 1300, 260),        # down: 22 of 96 tiles split, three parts each, then one whole tile per pair
    ("8b", 1700, 340),        # down: 38 of 112 tiles split over all pairs: parts cross the tiles
    ("deep-qkv", 1999, 1999), # q/k/v: all 24 tiles of the three matrices split; gate/up: 6 of 80, four parts each, then whole tiles
    ("deep-gate", 700, 140),  # gate/up: one tile of 75 split, four parts
]


@pytest.mark.parametrize("model,rows,states", SCHEDULES)
def test_schedules_of_the_products(model, rows, states):
    """Every row of a layer against the same rows in pieces of at most 128 (the persistent kernel, which the oracle checks at
    these shapes too), and three states against the oracle.  A bf16 operand is off by 2^-9 / sqrt(3) = 1.1e-3 (rms); each
    branch of the layer has two or three of those in a row, so a path is within about 3e-3 of the exact row and two paths
    within 4e-3 of each other; twice that is allowed (the deep models, whose branches outweigh the residual stream, use most of it)."""
    cfg = dataclasses.replace(DEEP.get(model) or datagen.CONFIGS[model], L=1, vocab=64)
    T, C = rows // states, 70
    p = Pair(cfg, max_ctx=C + T, max_rows=2048, max_M=1, max_T=1, gen_device="cuda")
    kv, ocache = p.new_kv(), p.new_oracle_cache()
    for t, k in ((kv.k, 0), (kv.v, 1)):
        t.copy_(datagen.normal_rows(64, k, tuple(t.shape)).to(cfg.torch_dtype))
    kv_to_oracle(kv, C + T, ocache)
    x = datagen.normal_rows(65, rows, (rows, cfg.d_model)).to(torch.float32)
    xd = x.cuda()
    got = p.engine.layer_forward(0, xd, states, T, C, C, kv)
    step = 128 // T
    pieces = [p.engine.layer_forward(0, xd[s * T:min(s + step, states) * T].contiguous(), min(step, states - s), T, C, C, kv)
              for s in range(0, states, step)]
    assert p.engine.device_status() == 0
    other = torch.cat(pieces)
    err = (got - other).norm(dim=1) / other.norm(dim=1)
    print(f"{model} {rows}: paths differ by {float(err.max()):.2e}", end=" ")
    assert float(err.max()) < 8e-3, int(err.argmax())
    g = got.cpu().numpy()
    for s in (0, states // 2, states - 1):
        rows_s = slice(s * T, (s + 1) * T)
        ref, _, _ = orc.decoder_layer(x[rows_s].double().numpy(), p.oracle.layer(0), ocache.k[0], ocache.v[0], C, C, cfg)
        e = np.linalg.norm(g[rows_s] - ref, axis=1) / np.linalg.norm(ref, axis=1)
        print(f"oracle {e.max():.2e}", end=" ")
        assert e.max() < 6e-3, (s, int(e.argmax()))
    p.engine.close()


@pytest.mark.parametrize("nq,nkv,R,C,sigma,delta", [
    (8, 2, 200, 700, 8.0, 0.25),     # four query heads per kv head, key splits
    (8, 2, 513, 190, 1.0, 0.5),      # few key tiles: no split
    (4, 4, 130, 1000, 4.0, 0.25),    # one query head per kv head
    (8, 1, 300, 333, 8.0, 0.25),     # eight
    (6, 2, 257, 130, 2.0, 0.5),      # three: rows straddle the blocks of 128 pairs
])
def test_attention_keeps_all_parts_of_its_operands(nq, nkv, R, C, sigma, delta):
    """The attention alone, out of a layer with W_o = 1 and W_down = 0 whose normed rows are +-1 (all exact in bf16):
    its result against float64, to the rounding of the bf16 operand that W_o reads (at most 2^-9 of a value) and an eighth
    of that for everything else.  Cached keys come in pairs that differ in one dim and carry opposite values, so weights
    cancel: with their low parts dropped the result is off by 0.8 - 4 %, with those of q by 0.3 - 0.8 %."""
    hd, dev = 128, "cuda"
    d = nq * hd
    cfg = dataclasses.replace(datagen.CONFIGS["mini8b"], name="attention", L=1, d_model=d, n_q_heads=nq, n_kv_heads=nkv, d_ffn=256,
                              vocab=64)
    g = torch.Generator(device=dev).manual_seed(nq * 1000 + R)

    def rnd(*shape, std=1.0):
        return (torch.randn(shape, device=dev, generator=g) * std).to(torch.bfloat16)

    def zero(*shape):
        return torch.zeros(shape, dtype=torch.bfloat16, device=dev)

    one = torch.ones(d, device=dev)
    kvd = nkv * hd
    # (keys of the rows themselves are zero: next to the cache's they weigh nothing, and their values are zero)
    lw = {"attn_norm": one, "wq": rnd(d, d, std=sigma / d ** 0.5), "wk": zero(kvd, d), "wv": zero(kvd, d),
          "wo": torch.eye(d, device=dev).to(torch.bfloat16), "mlp_norm": one, "w_gate": rnd(256, d), "w_up": rnd(256, d),
          "w_down": zero(d, 256)}
    ccfg = clasp.make_config(cfg, max_ctx=C + R, max_rows=R, max_M=1, max_T=1)
    e = clasp.Clasp(ccfg)
    e.load_layers(0, [lw])
    kv = clasp.KVCache(ccfg)
    k, v = rnd(C // 2, nkv, hd), rnd(C // 2, nkv, hd)
    k2 = k.clone()
    k2[:, :, 5] += delta
    n = C // 2 * 2                   # (the last key of an odd number: zero, with a zero value)
    kv.k[0, 0:n:2], kv.k[0, 1:n:2] = k, k2
    kv.v[0, 0:n:2], kv.v[0, 1:n:2] = v, -v
    x = torch.randint(0, 2, (R, d), device=dev, generator=g).float() * 2 - 1
    got = (e.layer_forward(0, x, 1, R, C, C, kv, write_kv=True) - x).double().view(R, nq, hd)
    assert e.device_status() == 0

    q = (x.double() @ lw["wq"].double().T).view(R, nq, hd)
    ang = (C + torch.arange(R, device=dev, dtype=torch.float64))[:, None] * cfg.rope_theta ** (
        -torch.arange(0, hd, 2, device=dev, dtype=torch.float64) / hd)
    cos, sin = ang.cos()[:, None], ang.sin()[:, None]
    q = torch.cat([q[..., :64] * cos - q[..., 64:] * sin, q[..., 64:] * cos + q[..., :64] * sin], -1)
    kk, vv = (t[0].double().repeat_interleave(nq // nkv, 1) for t in (kv.k, kv.v))
    s = torch.einsum("rhd,chd->hrc", q, kk) / hd ** 0.5
    s = s.masked_fill(torch.arange(C + R, device=dev)[None, None] > C + torch.arange(R, device=dev)[None, :, None], -torch.inf)
    want = torch.einsum("hrc,chd->rhd", s.softmax(-1), vv)
    err = float((got - want).norm() / want.norm())
    print(f"attention error {err:.6e}")
    assert err < 2.0 ** -9 * 1.125
    e.close()
