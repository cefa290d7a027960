"""Prefill attention over 128-slot KV tiles whose keys (and values) are NaN: a row
with a score above -inf in an earlier tile is NaN, tiles before its first such
score count as masked (their values still count times zero), and launches of whole
row tiles and of halves agree.  Other rows against attention in 64 bits."""
import math

import pytest
import torch

from wm_synth.device_problem import host_to_device
from wm_synth.inputs import prefill_queries

from . import _harness as H
from .test_gpu_prefill import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nan_v", [False, True])
@pytest.mark.parametrize("tiles", [(0,), (1,), (2,), (0, 1), (1, 2), (0, 2), (3,), (1, 3)])
@pytest.mark.parametrize("d,G,B,Hkv", [(64, 1, 1, 2), (96, 2, 1, 2), (128, 1, 1, 3), (96, 1, 8, 16), (64, 2, 8, 12)])
def test_nan_key_tiles(d, G, B, Hkv, tiles, nan_v):
    T, page = 600, 64  # five tiles
    w = _workload(d, G, page, T, B=B, Hkv=Hkv, L=1, k=1)
    prob, sess, dp = H.setup(w, seed=3, seq_lens=[T] * B)
    for b in range(B):
        for t in tiles:
            for lp in range(2 * t, 2 * t + 2):
                sess.k_pool[0, int(prob.page_table[b, lp])] = float("nan")
                if nan_v:
                    sess.v_pool[0, int(prob.page_table[b, lp])] = float("nan")
    q = host_to_device(prefill_queries(w, 5, B, T), "bf16", sess.device)
    pos = torch.arange(T, dtype=torch.int32, device=sess.device).repeat(B, 1)
    out = torch.full_like(q, 7.0)
    sess.prefill_attn(0, q, pos, dp.page_table, out)
    assert sess.read_status() == 0
    pages = dp.page_table[:, :(T + page - 1) // page].long()
    kv = [pool[0][pages].permute(0, 2, 1, 3, 4).reshape(B, Hkv, -1, d)[:, :, :T].double()
          for pool in (sess.k_pool, sess.v_pool)]
    K, V = (torch.nan_to_num(x, nan=0.0).repeat_interleave(G, 1) for x in kv)
    good = [t for t in range(5) if t not in tiles]
    tile = torch.arange(T, device=q.device) // 128
    first = good[0]
    scores = q.double().permute(0, 2, 1, 3) @ K.transpose(-1, -2) / math.sqrt(d)
    keep = (pos[0][None, :] <= pos[0][:, None]) & torch.isin(tile, torch.tensor(good, device=q.device))[None, :]
    want = (torch.softmax(scores.masked_fill(~keep, -math.inf), -1) @ V).permute(0, 2, 1, 3)
    for r0 in range(0, T, 128):  # rows r0 .. of row tile r0 / 128
        t, rows = r0 // 128, slice(r0, min(T, r0 + 128))
        after = any(first < x <= t for x in tiles)
        before = any(x < first and x <= t for x in tiles)
        if after or (before and nan_v):
            assert out[:, rows].isnan().all()
        elif t < first:
            assert not out[:, rows].any()
        else:
            assert H.rel_err(H.to_f64(out[:, rows]), want[:, rows].cpu().numpy()) <= H.TOL["bf16"]
    del sess, dp
    torch.cuda.empty_cache()
