"""Decode attention with several query heads per kv head (bf16): the stage
math on the tensor cores, in both kernels, against the fp64 oracle.

The sizes are the edges of its tiles: steps of 16 slots, stages of 16 or 32,
V in blocks of half a stage, pages smaller and larger than a block and a
stage, 32-column rest of d = 96."""
import pytest
import torch

from wm_synth import configs

from . import _harness as H

pytestmark = pytest.mark.gpu

# the rounding of the output to bf16's 8 significant bits (2^-8 at most) and the
# fp32 arithmetic before it (scores below 2^5 in log2 units, 128-term sums: below 2^-12)
TOL = 2.0**-8 + 2.0**-12
LENS = [1, 2, 15, 16, 17, 31, 33, 64, 700]


def _setup(d, G, page, **over):
    w = configs.Workload("t", L=2, k=2, D=64, Hq=2 * G, Hkv=2, d=d, B=len(LENS), ctx=700, ctx_lo=1,
                         page=page, dtype="bf16", chan_map="mod", permute_pages=True).with_(**over)
    return (w, *H.setup(w, seed=11, seq_lens=LENS))


def _run(sess, dp, w, layer, split):
    out = torch.full((w.B, w.Hq, w.d), float("nan"), dtype=sess.dtype, device=sess.device)
    kw = dict(unit_split=True) if split == "unit" else dict(dynamic_split=True)
    sess.decode_attn(layer, dp.q[layer], dp.page_table, dp.seq_lens, out, **kw)
    return out


@pytest.mark.parametrize("split", ["unit", "dynamic"])
@pytest.mark.parametrize("d,G,page", [
    (64, 4, 1), (64, 8, 4), (64, 4, 16), (64, 8, 64), (64, 2, 2), (64, 2, 32), (96, 2, 1), (96, 2, 16), (96, 2, 64), (96, 8, 2), (96, 4, 8), (96, 4, 128),
    (128, 8, 1), (128, 4, 4), (128, 8, 16), (128, 4, 32)])
def test_every_row(split, d, G, page):
    w, prob, sess, dp = _setup(d, G, page)
    for layer in range(w.L):
        got = H.to_f64(_run(sess, dp, w, layer, split))
        want = H.oracle_attn_full(prob, layer)
        assert H.rel_err(got, want) <= TOL, (layer, H.rel_err(got, want))
    assert sess.read_status() == 0


@pytest.mark.parametrize("split", ["unit", "dynamic"])
@pytest.mark.parametrize("d,G,page", [(64, 8, 16), (96, 2, 8), (96, 4, 16), (128, 4, 8), (128, 8, 64)])
def test_unwritten_slots_and_infinities(split, d, G, page):
    """NaN past a length changes no bit, a dummy-only sequence returns the
    dummy's value, and an infinite value reaches its own column alone."""
    w, prob, sess, dp = _setup(d, G, page, L=1, k=1)
    base = _run(sess, dp, w, 0, split).clone()
    pg = int(prob.page_table[0, 0])
    assert torch.equal(base[0], sess.v_pool[0, pg, :, 0, :].repeat_interleave(G, 0))
    for b, S in enumerate(LENS):
        for i in range(int((prob.page_table[b] >= 0).sum())):
            lo = max(0, S - i * page)
            if lo < page:
                p = int(prob.page_table[b, i])
                sess.k_pool[:, p, :, lo:, :] = float("nan")
                sess.v_pool[:, p, :, lo:, :] = float("nan")
    assert torch.equal(_run(sess, dp, w, 0, split), base)
    for b, col in ((4, 0), (5, d - 1)):
        sess.v_pool[0, int(prob.page_table[b, 0]), 1, 0, col] = float("inf")
    got = _run(sess, dp, w, 0, split)
    want = base.clone()
    want[4, G:, 0] = float("inf")
    want[5, G:, d - 1] = float("inf")
    assert torch.equal(got, want)
    assert sess.read_status() == 0
