"""One decoder layer over more rows than the skinny products take (the tensor-core products and attention of
csrc/wide.cuh) against the oracle: edges of the 256-row and 256-feature tiles, ragged key tiles, several states with
their own rows only, key splits, and a row maximum that moves in mid-cache (the rescaling path)."""
import ctypes

import numpy as np
import pytest
import torch

import datagen
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
