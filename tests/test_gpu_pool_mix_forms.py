"""The pool's bf16 mix in both its forms: a CTA per token (or part of one) with
channels and layers that do not fill their blocks of 16, and a warp per token from
768 tokens (17 to 32 layers) or 1536 on; the prenorm's rows of two warps, an odd
number of them."""
import pytest
import torch

from . import _harness as H
from .test_gpu_pool_mix import _w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,k,D,B,p", [
    (16, 16, 72, 300, 2), (20, 5, 328, 257, 2), (33, 2, 72, 180, 3),
    (5, 3, 1032, 1, 1), (7, 5, 2048, 9, 2), (9, 9, 1544, 65, 4), (21, 18, 2056, 3, 2)])
def test_pool_mix_cta_form(L, k, D, B, p):
    """Every written key and value against the fp64 oracle."""
    prob, sess, dp = H.setup(_w(L, k, D, B, p, Hkv=1), seed=7)
    sess.kv_mix(dp.h, dp.page_table, dp.slot)
    torch.cuda.synchronize()
    assert sess.read_status() == 0
    want = H.oracle_mix_tokens(prob)
    got = {bj: H.gpu_written_kv(sess, prob, *bj) for bj in want}
    for i in (0, 1):
        assert max(H.rel_err(got[bj][i], want[bj][i]) for bj in want) <= H.TOL["bf16"]
    torch.cuda.empty_cache()


@pytest.mark.parametrize("L,k,D,B,p", [
    (3, 2, 136, 1537, 1), (16, 16, 72, 1536, 2), (20, 5, 328, 769, 2), (32, 17, 64, 768, 4),
    (33, 3, 64, 1538, 3), (40, 2, 1096, 1600, 2)])
def test_pool_mix_warp_form(L, k, D, B, p):
    """The same tokens in calls of 60 (the CTA form, checked against the oracle):
    operands, states and sums are the same but for the order of fp32 sums, so an
    output differs by its own rounding to bf16 (one step, 2^-8) and by what an
    operand element rounded the other way makes of one of D products: 2^-7 of the
    head's largest covers both."""
    prob, sess, dp = H.setup(_w(L, k, D, B, p, Hkv=1), seed=7)
    sess.kv_mix(dp.h, dp.page_table, dp.slot)
    whole = [x.clone().float() for x in (sess.k_pool, sess.v_pool)]
    sess.k_pool.zero_()
    sess.v_pool.zero_()
    for b in range(0, B, 60):
        t = slice(b, min(B, b + 60))
        sess.kv_mix(dp.h[t].contiguous(), dp.page_table[t].contiguous(), dp.slot[t].contiguous(), B=t.stop - b)
    torch.cuda.synchronize()
    assert sess.read_status() == 0
    slot = dp.slot.long()
    page = dp.page_table[torch.arange(B, device=slot.device), slot // prob.w.page].long()
    for big, pool in zip(whole, (sess.k_pool, sess.v_pool)):
        a, c = (x[:, page, :, slot % prob.w.page].float() for x in (big, pool))  # [B][k][1][d]
        assert c.abs().amax(-1).min() > 0
        assert ((a - c).abs().amax(-1) <= 2.0 ** -7 * c.abs().amax(-1)).all()
    del sess, dp
    torch.cuda.empty_cache()
