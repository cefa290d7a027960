"""The prefill attention's work items (wm_prefill_attn): more items than SMs,
so that every CTA takes several; query tiles of unequal extent and rows that
see nothing; and scores that keep growing along the slots, so that running
maxima are raised (and O rescaled) in many steps.  Every row against the fp64
oracle."""
import numpy as np
import pytest
import torch

from wm_synth.inputs import prefill_queries

from . import _harness as H
from .test_gpu_prefill import _oracle, _run, _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,G,page,B,Hkv,T,q_scale", [
    (128, 1, 16, 8, 16, 385, 1.0),    # 256 items of two row tiles, the last one ragged
    (96, 2, 8, 8, 8, 300, 64.0),      # 192 items of head pairs, maxima raised at every tile
    (64, 4, 32, 16, 4, 257, 64.0),    # 384 items, one row in the last tile
    (128, 1, 128, 5, 16, 640, 64.0),
])
def test_prefill_items_match_oracle(d, G, page, B, Hkv, T, q_scale):
    w = _workload(d, G, page, T, B=B, Hkv=Hkv, L=1, k=1).with_(q_scale=q_scale)
    prob, sess, dp = H.setup(w, seed=12, seq_lens=[T] * B)
    pos = np.stack([np.arange(T, dtype=np.int32)] * B)
    # one sequence whose rows see short extents in the second tile only, one
    # whose first tile sees nothing (bad positions: zero rows)
    pos[0, 128:] = pos[0, 128:] % 40
    pos[1, :128] = -1
    q_bits = prefill_queries(w, 91, B, T)
    got = _run(sess, q_bits, pos, dp, 0)
    assert sess.read_status() == 4  # WM_ERR_BOUNDS: the bad positions
    assert torch.count_nonzero(got[1, :128].float()) == 0
    units = [(b, r, h) for b in range(B) for r in range(T) for h in range(w.Hq)
             if pos[b, r] >= 0 and (b < 2 or (r * 7 + h) % 5 == 0 or r in (0, 127, 128, T - 1))]
    want = _oracle(prob, q_bits, np.maximum(pos, 0), 0, units=units)
    idx = torch.tensor(units, device=got.device)
    gotv = H.to_f64(got[idx[:, 0], idx[:, 1], idx[:, 2]])
    assert H.rel_err(gotv, want) <= H.TOL["bf16"]
    del sess, dp
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
