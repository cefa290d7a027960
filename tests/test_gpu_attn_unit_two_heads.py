"""Unit split with two query heads of 64 per kv head (bf16): the stage math runs on
the tensor cores with pages of at most 16 slots or room for at most 2048, else on the
CUDA cores.  Both sides of each line against the fp64 oracle."""
import pytest
import torch

from paper_2608_18486_gb300 import _lib as W
from wm_synth import configs

from . import _harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("page,slots", [(16, 2064), (32, 2048), (32, 2080), (1, 2049), (64, 2112), (8, 304), (128, 5120)])
def test_both_sides(page, slots):
    lens = [slots - 1, 1, 33, slots // 2, 777 % slots, 16]
    w = configs.Workload("t", L=1, k=1, D=64, Hq=6, Hkv=3, d=64, B=len(lens), ctx=slots, page=page,
                         dtype="bf16", chan_map="mod", permute_pages=True)
    prob, sess, dp = H.setup(w, seed=9, seq_lens=lens)
    assert prob.max_pages * page == slots
    assert W.wm_decode_attn_plan(sess.cfg, w.B, prob.max_pages, 0)["unit_ctas"] > 0
    got = H.to_f64(H.run_attn(sess, dp, 0))
    assert H.rel_err(got, H.oracle_attn_full(prob, 0)) <= H.TOL["bf16"]
    assert sess.read_status() == 0
    torch.cuda.empty_cache()
