"""Prefill attention of sequences with room for one KV tile (128 slots): few items,
but nothing for a CTA's halves to share, so the launch takes whole tiles.  The same
rows with room for more slots, where it takes halves, and against the fp64 oracle."""
import numpy as np
import pytest
import torch

from wm_synth.device_problem import host_to_device
from wm_synth.inputs import prefill_queries

from . import _harness as H
from .test_gpu_prefill import _oracle, _run, _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,G,page,T", [
    (64, 1, 16, 1), (96, 2, 8, 40), (128, 4, 128, 127), (64, 2, 64, 127), (96, 1, 32, 100), (128, 1, 16, 64)])
def test_one_kv_tile(d, G, page, T):
    w = _workload(d, G, page, T, L=1, k=1)
    prob, sess, dp = H.setup(w, seed=43, seq_lens=[T, T])
    assert prob.max_pages * page <= 128
    pos = np.stack([np.arange(T, dtype=np.int32), np.arange(T, dtype=np.int32)[::-1]])
    q_bits = prefill_queries(w, 29, w.B, T)
    got = _run(sess, q_bits, pos, dp, 0)
    assert sess.read_status() == 0
    assert H.rel_err(H.to_f64(got), _oracle(prob, q_bits, pos, 0)) <= H.TOL["bf16"]
    # a page table of more than 128 slots, its further pages not there: the second
    # half is idle, the merge multiplies by 1 and adds 0
    wide = 128 // page + 1
    table = torch.full((w.B, wide), -1, dtype=torch.int32, device=sess.device)
    table[:, :prob.max_pages] = dp.page_table
    sess.max_pages = wide
    out = torch.empty_like(got)
    sess.prefill_attn(0, host_to_device(q_bits, "bf16", sess.device),
                      torch.from_numpy(np.ascontiguousarray(pos)).to(sess.device), table, out)
    torch.cuda.synchronize()
    assert sess.read_status() == 0
    assert torch.equal(out, got)
    torch.cuda.empty_cache()
