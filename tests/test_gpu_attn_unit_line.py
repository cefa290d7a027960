"""The planner's line for four-warp unit-split CTAs (bf16, four or eight query heads
per kv head, more units than SMs): by the bytes one unit has room for, since one CTA
streams the longest unit alone.  Both sides of it against the oracle, with one
sequence of full length among short ones."""
import pytest
import torch

from paper_2608_18486_gb300 import _lib as W
from wm_synth import configs

from . import _harness as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,G,slots,unit", [
    (64, 4, 2336, True), (64, 4, 2352, False), (128, 8, 1168, True), (128, 8, 1184, False)])
def test_unit_line(d, G, slots, unit):
    w = configs.Workload("t", L=1, k=1, D=64, Hq=8 * G, Hkv=8, d=d, B=24, ctx=slots, page=16, dtype="bf16",
                         chan_map="mod", permute_pages=True)
    prob, sess, dp = H.setup(w, seed=5, seq_lens=[30] * 4 + [slots - 1] + [17] * 19)
    assert prob.max_pages * w.page == slots
    assert (W.wm_decode_attn_plan(sess.cfg, w.B, prob.max_pages, 0)["unit_ctas"] > 0) == unit
    got = H.to_f64(H.run_attn(sess, dp, 0))
    assert H.rel_err(got, H.oracle_attn_full(prob, 0)) <= H.TOL["bf16"]
    assert sess.read_status() == 0
    torch.cuda.empty_cache()
