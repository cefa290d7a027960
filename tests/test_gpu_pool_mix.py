"""The pool's mix (Sec. 3.1 Steps 1-2) at the edges of its tensor-core tiling:
layers past one and two blocks of 16, channels past 16, D that is not a
multiple of a warp's 64 elements, one token and groups around the batched
threshold.  Every written key and value against the fp64 oracle."""
import pytest
import torch

from paper_2608_18486_gb300 import _lib as W
from wm_synth import configs

from . import _harness as H

pytestmark = pytest.mark.gpu


def _w(L, k, D, B, p=2, Hkv=2, d=64):
    return configs.Workload("mix", L=L, k=k, D=D, Hq=Hkv, Hkv=Hkv, d=d, B=B, ctx=40, page=16,
                            dtype="bf16", chan_map="mod", ctx_lo=1, permute_pages=True, p=p,
                            gain_std=0.1)


@pytest.mark.parametrize("L,k,D,B,p", [
    (16, 16, 64, 1, 2), (17, 16, 72, 3, 2), (32, 17, 328, 5, 1), (33, 33, 72, 2, 3),
    (40, 20, 200, 70, 2), (16, 1, 520, 64, 2), (20, 5, 1032, 63, 2), (3, 3, 136, 129, 1),
    (32, 8, 4096, 65, 4)])
def test_pool_mix_edges(L, k, D, B, p):
    prob, sess, dp = H.setup(_w(L, k, D, B, p), seed=4)
    sess.k_pool.fill_(float("nan"))
    sess.v_pool.fill_(float("nan"))
    sess.kv_mix(dp.h, dp.page_table, dp.slot)
    torch.cuda.synchronize()
    assert sess.read_status() == 0
    want = H.oracle_mix_tokens(prob)
    errk = max(H.rel_err(H.gpu_written_kv(sess, prob, b, j)[0], want[b, j][0]) for b, j in want)
    errv = max(H.rel_err(H.gpu_written_kv(sess, prob, b, j)[1], want[b, j][1]) for b, j in want)
    assert errk <= H.TOL["bf16"] and errv <= H.TOL["bf16"], (errk, errv)
    # nothing but the addressed slots was written
    written = sum(int((~torch.isnan(t.float())).sum()) for t in (sess.k_pool, sess.v_pool))
    w = prob.w
    assert written == 2 * w.B * w.k * w.Hkv * w.d
    torch.cuda.empty_cache()
