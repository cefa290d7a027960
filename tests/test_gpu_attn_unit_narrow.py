"""Decode attention with more (sequence, kv head) units than SMs and four or
eight bf16 query heads per kv head: the unit split in CTAs of four warps, two
per SM, up to the line where launches stream.  Every row against the oracle."""
import numpy as np
import pytest
import torch

from paper_2608_18486_gb300 import _lib as W
from wm_synth import configs

from . import _harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,G,B,ctx,warps", [
    (64, 8, 25, 300, 4), (96, 4, 32, 130, 4), (128, 4, 25, 65, 4), (128, 8, 37, 200, 4),
    (64, 4, 19, 300, 8), (64, 4, 64, 40, None)])  # 152 units fit 8 warps each; 512 fit neither way
def test_many_units_every_row(d, G, B, ctx, warps):
    w = configs.Workload("t", L=1, k=1, D=64, Hq=8 * G, Hkv=8, d=d, B=B, ctx=ctx, ctx_lo=1, page=16,
                         dtype="bf16", chan_map="mod", permute_pages=True)
    lens = np.random.default_rng(3).integers(1, ctx + 1, B)
    lens[:2] = 1, ctx
    prob, sess, dp = H.setup(w, seed=5, seq_lens=[int(s) for s in lens])
    plan = W.wm_decode_attn_plan(sess.cfg, B, prob.max_pages, 0)
    if warps is None or plan["unit_ctas"] == 0:
        assert warps != 4 and plan["unit_ctas"] == 0, plan
    else:
        assert plan["warps"] == plan["grid"] * warps and plan["grid"] == 8 * B * plan["unit_ctas"], plan
    got = H.to_f64(H.run_attn(sess, dp, 0))
    assert H.rel_err(got, H.oracle_attn_full(prob, 0)) <= H.TOL["bf16"]
    assert sess.read_status() == 0
    torch.cuda.empty_cache()
