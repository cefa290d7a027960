"""The pool over groups of tokens (Sec. 3.3 passes; 128 tokens and more take the
tokens as MMA rows): every written key and value against the fp64 oracle at the
edges of the tiles -- token tiles of one row and of all rows, heads that leave a
unit half full, channels of several tiles, logits that are not a multiple of
four or span two tiles, D of a partial k-block -- bad slots and pages skipped
and reported, and a key-norm gain that is not 16-byte aligned."""
import pytest
import torch

from paper_2608_18486_gb300 import _lib as W
from wm_synth import configs

from . import _harness as H

pytestmark = pytest.mark.gpu


def _setup(L, k, D, B, Hkv, d, page=16):
    w = configs.Workload("rows", L=L, k=k, D=D, Hq=Hkv, Hkv=Hkv, d=d, B=B, ctx=40, page=page,
                         dtype="bf16", chan_map="mod", ctx_lo=1, permute_pages=True, gain_std=0.1)
    return H.setup(w, seed=6)


def _check(prob, sess, skip=()):
    want = H.oracle_mix_tokens(prob)
    keep = [bj for bj in want if bj[0] not in skip]
    errk = max(H.rel_err(H.gpu_written_kv(sess, prob, b, j)[0], want[b, j][0]) for b, j in keep)
    errv = max(H.rel_err(H.gpu_written_kv(sess, prob, b, j)[1], want[b, j][1]) for b, j in keep)
    assert errk <= H.TOL["bf16"] and errv <= H.TOL["bf16"], (errk, errv)


@pytest.mark.parametrize("L,k,D,B,Hkv,d", [
    (5, 3, 128, 128, 3, 64),     # a unit of one head, 15 logits
    (7, 5, 72, 129, 4, 96),      # units 3 + 1, one token in the second tile, partial k-block
    (20, 16, 64, 300, 3, 128),   # 320 logits, tiles of 2 + 1 units
    (4, 4, 512, 255, 1, 96), (16, 16, 320, 384, 5, 64), (3, 2, 1024, 640, 2, 128)])
def test_pool_rows_edges(L, k, D, B, Hkv, d):
    prob, sess, dp = _setup(L, k, D, B, Hkv, d)
    assert W.wm_kv_mix_launches(sess.cfg, B) == 4
    sess.k_pool.fill_(float("nan"))
    sess.v_pool.fill_(float("nan"))
    sess.kv_mix(dp.h, dp.page_table, dp.slot)
    torch.cuda.synchronize()
    assert sess.read_status() == 0
    _check(prob, sess)
    written = sum(int((~torch.isnan(t.float())).sum()) for t in (sess.k_pool, sess.v_pool))
    assert written == 2 * B * k * Hkv * d
    k1, v1 = sess.k_pool.clone(), sess.v_pool.clone()
    sess.kv_mix(dp.h, dp.page_table, dp.slot)  # the same bits again
    torch.cuda.synchronize()
    assert torch.equal(k1.view(torch.int16), sess.k_pool.view(torch.int16))
    assert torch.equal(v1.view(torch.int16), sess.v_pool.view(torch.int16))
    torch.cuda.empty_cache()


def test_pool_rows_bad_slots_and_unaligned_gain():
    prob, sess, dp = _setup(4, 3, 192, 160, 3, 96)
    # a gain two bytes past a 16-byte boundary: the decode form of the projection
    qk = torch.empty(dp.qk_g.numel() + 1, dtype=dp.qk_g.dtype, device=dp.qk_g.device)
    qk[1:] = dp.qk_g.reshape(-1)
    ws = list(dp.weights())
    ws[5] = qk[1:].view(dp.qk_g.shape)
    for weights in (dp.weights(), tuple(ws)):
        sess.set_weights(*weights)
        sess.k_pool.fill_(float("nan"))
        sess.v_pool.fill_(float("nan"))
        slot = dp.slot.clone()
        slot[7] = 0                                # the dummy's slot
        slot[130] = prob.max_pages * prob.w.page   # past the table
        pt = dp.page_table.clone()
        pt[128, int(prob.seq_lens[128]) // prob.w.page] = prob.num_pages
        sess.kv_mix(dp.h, pt, slot)
        torch.cuda.synchronize()
        assert sess.read_status() == W.WM_ERR_BOUNDS
        _check(prob, sess, skip=(7, 128, 130))
        written = int((~torch.isnan(sess.k_pool.float())).sum())
        assert written == 157 * prob.w.k * prob.w.Hkv * prob.w.d
    torch.cuda.empty_cache()
