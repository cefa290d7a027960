"""Prefill attention launches of few items (wm_prefill_attn), where a CTA's two
halves share out one row tile's KV tiles: one, two and odd numbers of KV
tiles, a row past a tile's edge, rows that see nothing, maxima that keep
growing, and CTAs that take several items.  Every row (or a sample of the
large case) against the fp64 oracle."""
import numpy as np
import pytest
import torch

from wm_synth.inputs import prefill_queries

from . import _harness as H
from .test_gpu_prefill import _oracle, _oracle_units, _run, _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,G,page,T,q_scale", [
    (64, 1, 16, 1, 1.0), (96, 2, 8, 127, 64.0), (128, 4, 64, 128, 1.0), (96, 1, 128, 129, 64.0),
    (128, 1, 16, 256, 64.0), (64, 8, 256, 257, 1.0), (128, 2, 32, 513, 64.0)])
def test_halves_match_oracle(d, G, page, T, q_scale):
    w = _workload(d, G, page, T, L=1, k=1).with_(q_scale=q_scale)
    prob, sess, dp = H.setup(w, seed=31, seq_lens=[T, T])
    pos = np.stack([np.arange(T, dtype=np.int32)] * w.B)
    bad = T // 2 if T > 1 else None
    if bad:
        pos[1, bad] = -1
    q_bits = prefill_queries(w, 17, w.B, T)
    got = H.to_f64(_run(sess, q_bits, pos, dp, 0))
    want = _oracle(prob, q_bits, np.maximum(pos, 0), 0)
    if bad:
        assert sess.read_status() == 4  # WM_ERR_BOUNDS, and zero rows
        assert not got[1, bad].any()
        want[1, bad] = 0.0
    assert H.rel_err(got, want) <= H.TOL["bf16"]
    torch.cuda.empty_cache()


def test_halves_over_several_items_per_cta():
    T = 1700  # 336 items of one 128-row tile
    w = _workload(96, 1, 16, T, B=4, Hkv=6, L=1, k=1)
    prob, sess, dp = H.setup(w, seed=32, seq_lens=[T] * 4)
    pos = np.stack([np.arange(T, dtype=np.int32)] * w.B)
    q_bits = prefill_queries(w, 18, w.B, T)
    got = _run(sess, q_bits, pos, dp, 0)
    units = [(b, r, h) for b in range(w.B) for h in range(w.Hq) for r in range(b + h, T, 67)]
    idx = torch.tensor(units, device=got.device)
    gotv = H.to_f64(got[idx[:, 0], idx[:, 1], idx[:, 2]])
    assert H.rel_err(gotv, _oracle_units(prob, q_bits, pos, 0, units)) <= H.TOL["bf16"]
    assert sess.read_status() == 0
    torch.cuda.empty_cache()
