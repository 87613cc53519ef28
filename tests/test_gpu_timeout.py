"""The wind-down path of the kernels' bounded waits, reached without a kernel that would wait
forever: the context's wait limit is set to one poll, so the first wait of a healthy launch that is
not satisfied at once (a copy still in flight) gives up.  The kernel must then end by itself (copies
in flight awaited, tensor memory freed), the status call must report CLASP_ERR_TIMEOUT once, and the
context must work again after the limit is restored."""
import dataclasses

import pytest
import torch

import datagen
from oracle import clasp_oracle as orc
from tests.util import Pair, close_hidden, kv_to_oracle, tol_hidden

pytestmark = pytest.mark.gpu

TIMEOUT = -6


@pytest.fixture(scope="module")
def pair():
    cfg = datagen.CONFIGS["small"]
    p = Pair(cfg, max_ctx=96, max_rows=32, max_M=2, max_T=1, max_head_rows=4)
    yield p
    p.engine.close()


def _layer_inputs(pair):
    cfg = pair.cfg
    kv = pair.new_kv()
    kv.k.copy_(datagen.normal_rows(81, 0, tuple(kv.k.shape)).to(cfg.torch_dtype))
    kv.v.copy_(datagen.normal_rows(81, 1, tuple(kv.v.shape)).to(cfg.torch_dtype))
    x = datagen.normal_rows(82, 0, (4, cfg.d_model)).to(torch.float32)
    return kv, x


def test_gemm_wait_that_runs_out_is_reported_and_the_context_recovers(pair):
    eng = pair.engine
    x = datagen.normal_rows(83, 0, (5, 1376)).to(torch.bfloat16).cuda()
    w = datagen.normal_rows(83, 1, (1000, 1376), 0.05).to(torch.bfloat16).cuda()
    good = eng.gemm_xwT(x, w)
    assert eng.device_status() == 0
    eng.set_wait_limit(1)
    eng.gemm_xwT(x, w)
    assert eng.device_status() == TIMEOUT
    assert eng.device_status() == 0            # reported once, then cleared
    eng.set_wait_limit(0)
    again = eng.gemm_xwT(x, w)
    assert eng.device_status() == 0
    assert torch.equal(again, good)


def test_layer_kernel_wait_that_runs_out_is_reported_and_the_context_recovers(pair):
    cfg, eng = pair.cfg, pair.engine
    assert eng.engine_active()
    kv, x = _layer_inputs(pair)
    good = eng.layer_forward(2, x.cuda(), 4, 1, 40, 40, kv)
    assert eng.device_status() == 0
    eng.set_wait_limit(1)
    eng.layer_forward(2, x.cuda(), 4, 1, 40, 40, kv)
    assert eng.device_status() == TIMEOUT
    assert eng.device_status() == 0
    eng.set_wait_limit(0)
    again = eng.layer_forward(2, x.cuda(), 4, 1, 40, 40, kv)
    assert eng.device_status() == 0
    assert torch.equal(again, good)
    # and the recovered context still computes the layer: one state against the oracle
    ocache = pair.new_oracle_cache()
    kv_to_oracle(kv, pair.max_ctx, ocache)
    ref, _, _ = orc.decoder_layer(x[:1].double().numpy(), pair.oracle.layer(2), ocache.k[2], ocache.v[2], 40, 40, cfg)
    assert close_hidden(again[:1].cpu().numpy(), ref, tol_hidden(cfg))


@pytest.mark.parametrize("n", [129, 700])
def test_many_row_kernels_whose_waits_run_out_are_reported_and_the_context_recovers(n):
    """Layers over more than 128 rows (products with and without split tiles, attention): every launch of the call gives up."""
    cfg = datagen.CONFIGS["mini8b"]
    p = Pair(cfg, max_ctx=1024, max_rows=700, max_M=1, max_T=1, max_head_rows=4)
    eng = p.engine
    toks = datagen.token_ids(cfg, n).to(torch.int32).cuda()
    kv = p.new_kv()
    _, good = eng.verify(toks, 300, kv, 1)
    assert eng.device_status() == 0
    for polls in (1, 3, 20):                       # moderate limits: some waits succeed, others run out
        eng.set_wait_limit(polls)
        eng.verify(toks, 300, p.new_kv(), 1)
        status = eng.device_status()
        assert status == TIMEOUT if polls == 1 else status in (0, TIMEOUT)
        assert eng.device_status() == 0
    eng.set_wait_limit(0)
    _, again = eng.verify(toks, 300, kv, 1)
    assert eng.device_status() == 0
    assert torch.equal(again, good)
    eng.close()


def test_one_cluster_kernel_under_the_shortest_limit_ends_and_the_context_recovers():
    """The fp32 kernel of a whole call.  Its weight slices are fetched before the first rows are ready and then a layer
    ahead, so that even a limit of one poll is hardly ever reached on a healthy launch: the status may be either, the call
    ends and the context computes the same bits afterwards.  (That the call winds down when a wait does run out is shown
    by reading: the thread that gave up arms no barrier again, the other hand-offs are barriers that all threads reach.)"""
    cfg = dataclasses.replace(datagen.CONFIGS["tiny"], name="large-slices", L=4, d_model=384, n_q_heads=8, n_kv_heads=8, d_ffn=16)
    p = Pair(cfg, max_ctx=64, max_rows=16, max_M=2, max_T=1, max_head_rows=4)
    eng = p.engine
    toks = datagen.token_ids(cfg, 3).to(torch.int32).cuda()
    kv = p.new_kv()
    n0 = eng.launch_count()
    _, good = eng.verify(toks, 20, kv, 0)
    assert eng.launch_count() - n0 == 1
    s_good = eng.dp_search(good[2], cfg.d_model, 0, kv, 22, 22, 1, 2)
    assert eng.device_status() == 0
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    eng.set_wait_limit(1)
    for _ in range(4):
        flush.zero_()                               # (the weights come from memory, not from L2)
        eng.verify(toks, 20, p.new_kv(), 0)
        assert eng.device_status() in (0, TIMEOUT)
        eng.dp_search(good[2], cfg.d_model, 0, kv, 22, 22, 1, 2)
        assert eng.device_status() in (0, TIMEOUT)
        assert eng.device_status() == 0
    eng.set_wait_limit(0)
    _, again = eng.verify(toks, 20, kv, 0)
    s_again = eng.dp_search(good[2], cfg.d_model, 0, kv, 22, 22, 1, 2)
    assert eng.device_status() == 0
    assert torch.equal(again, good) and torch.equal(s_again["S"], s_good["S"])
    assert torch.equal(s_again["g_final"], s_good["g_final"])
    eng.close()
