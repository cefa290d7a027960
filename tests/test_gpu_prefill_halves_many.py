"""Prefill attention launches that take one row tile per item, its KV tiles shared
out over a CTA's halves, and have more items than SMs: sums, outputs, barriers and
ring slots carry over from item to item.  Causal rows, strided ones (a partial last
KV tile in every item) and items of one to five KV tiles in any order (the second
half idle in some), one position out of range.  A sample of the rows against the
fp64 oracle."""
import numpy as np
import pytest
import torch

from wm_synth.inputs import prefill_queries

from . import _harness as H
from .test_gpu_prefill import _oracle_units, _run, _workload

pytestmark = pytest.mark.gpu


def _items(Tq, B, Hq, G):
    """Items of a halves launch, and whether the launcher takes that form."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    pair = G % 2 == 0
    nblk = -(-Tq // (128 if pair else 256))
    whole = nblk * B * (Hq // 2 if pair else Hq)
    return -(-Tq // 128) * B * Hq, whole * (nblk + 1) / (2 * nblk) < 0.4 * sms, sms


@pytest.mark.parametrize("d,G,page,B,Hkv,Tq", [
    (64, 1, 16, 1, 12, 2040), (96, 2, 32, 2, 3, 2100), (128, 1, 64, 1, 6, 4500), (64, 8, 64, 1, 2, 1700)])
@pytest.mark.parametrize("rows", ["causal", "strided", "mixed"])
def test_many_halves_items(d, G, page, B, Hkv, Tq, rows):
    items, halves, sms = _items(Tq, B, Hkv * G, G)
    assert halves and items > sms
    rng = np.random.default_rng(d + G)
    if rows == "mixed":
        T = 600
        ext = np.repeat(rng.choice([1, 40, 128, 129, 255, 300, 400, 600], (B, Tq // 128 + 1)), 128, axis=1)[:, :Tq]
        pos = (rng.random((B, Tq)) * ext).astype(np.int32)
    else:
        step = 2 if rows == "strided" else 1
        T = step * Tq
        pos = np.stack([np.arange(step - 1, T, step, dtype=np.int32)] * B)
    w = _workload(d, G, page, T, B=B, Hkv=Hkv, L=1, k=1).with_(q_scale=8.0)
    prob, sess, dp = H.setup(w, seed=33, seq_lens=[T] * B)
    pos[0, 700] = -1
    q_bits = prefill_queries(w, 19, B, Tq)
    got = _run(sess, q_bits, pos, dp, 0)
    assert sess.read_status() == 4 and not got[0, 700].any()  # WM_ERR_BOUNDS
    units = [(b, r, h) for b in range(B) for h in range(w.Hq) for r in range(b + h, Tq, 101) if pos[b, r] >= 0]
    idx = torch.tensor(units, device=got.device)
    gotv = H.to_f64(got[idx[:, 0], idx[:, 1], idx[:, 2]])
    assert H.rel_err(gotv, _oracle_units(prob, q_bits, pos, 0, units)) <= H.TOL["bf16"]
    assert torch.isfinite(got.float()).all()
    # the same call again, into other memory: the same bits
    assert torch.equal(_run(sess, q_bits, pos, dp, 0).view(torch.int16), got.view(torch.int16))
    del sess, dp
    torch.cuda.empty_cache()
