"""The fp32 pool of a small decode batch (Sec. 3.1 Steps 1-2): the products
that stream the weights for at most sixteen tokens, on both sides of its lines,
with odd rows, reductions shorter than a warp's step and splits that end in
the middle of one.  Every written key and value against the fp64 oracle."""
import pytest
import torch

from wm_synth import configs

from . import _harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,k,D,Hkv,d,B,p", [
    (1, 1, 8, 1, 64, 1, 1), (3, 3, 72, 1, 96, 2, 2), (7, 5, 264, 3, 96, 3, 2), (16, 16, 512, 3, 96, 4, 2),
    (5, 3, 1032, 2, 128, 5, 1), (9, 9, 520, 4, 64, 8, 3), (9, 9, 520, 4, 64, 9, 3),
    (7, 5, 264, 3, 96, 16, 2), (3, 3, 72, 1, 96, 17, 2)])
def test_pool_f32_few_tokens(L, k, D, Hkv, d, B, p):
    w = configs.Workload("f32", L=L, k=k, D=D, Hq=Hkv, Hkv=Hkv, d=d, B=B, ctx=40, page=16, dtype="f32",
                         chan_map="mod", ctx_lo=1, permute_pages=True, p=p, gain_std=0.1)
    prob, sess, dp = H.setup(w, seed=4)
    sess.kv_mix(dp.h, dp.page_table, dp.slot)
    torch.cuda.synchronize()
    assert sess.read_status() == 0
    want = H.oracle_mix_tokens(prob)
    for X in (0, 1):
        err = max(H.rel_err(H.gpu_written_kv(sess, prob, b, j)[X], want[b, j][X]) for b, j in want)
        assert err <= H.TOL["f32"], (X, err)
