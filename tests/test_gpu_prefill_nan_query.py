"""Prefill attention: a query row of NaN gives a row of zeros and changes no bit
of any other row, in launches of whole row tiles and of halves."""
import pytest
import torch

from wm_synth.device_problem import host_to_device
from wm_synth.inputs import prefill_queries

from . import _harness as H
from .test_gpu_prefill import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,G,B,Hkv,T", [(96, 2, 2, 2, 300), (64, 1, 1, 1, 129), (128, 1, 8, 16, 385)])
def test_nan_queries(d, G, B, Hkv, T):
    w = _workload(d, G, 16, T, B=B, Hkv=Hkv, L=1, k=1)
    prob, sess, dp = H.setup(w, seed=9, seq_lens=[T] * B)
    q = host_to_device(prefill_queries(w, 5, B, T), "bf16", sess.device)
    pos = torch.arange(T, dtype=torch.int32, device=sess.device).repeat(B, 1)
    base = torch.empty_like(q)
    sess.prefill_attn(0, q, pos, dp.page_table, base)
    rows = [0, 37, 128, T - 1]
    q[:, rows] = float("nan")
    out = torch.full_like(q, float("nan"))
    sess.prefill_attn(0, q, pos, dp.page_table, out)
    base[:, rows] = 0
    assert torch.equal(out, base)
    assert sess.read_status() == 0
