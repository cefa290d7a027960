"""Prefill attention over batches of short prompts (wm_prefill_attn): more items
than SMs, nearly all of them with a partial last KV tile, so that the V tiles of
several items of one CTA are in the ring at once and each one's rows past the last
slot are zeroed before it is used.  Every row against the fp64 oracle."""
import numpy as np
import pytest
import torch

from wm_synth.inputs import prefill_queries

from . import _harness as H
from .test_gpu_prefill import _oracle, _run, _workload

pytestmark = pytest.mark.gpu

EXTENTS = {"one": [40], "two": [129, 200, 255], "mixed": [40, 127, 129, 200, 255, 500]}


@pytest.mark.parametrize("d,G,page", [(64, 1, 16), (64, 2, 8), (96, 1, 32), (96, 2, 16), (128, 1, 64), (128, 2, 16)])
@pytest.mark.parametrize("extents", ["one", "two", "mixed", "strided"])
def test_short_prompts_match_oracle(d, G, page, extents):
    B, Hkv = 64, 3  # 192 items of two row tiles of a head, or of a head pair
    if extents == "strided":  # every other position: a row block of two partial tiles, one of four
        lens = np.full(B, 500)
        pos = np.stack([np.arange(0, 500, 2)] * B)
    else:
        lens = np.random.default_rng(d + G).choice(EXTENTS[extents], B)
        pos = np.stack([np.arange(max(0, n - 130), max(0, n - 130) + 130) % n for n in lens])
    pos = pos.astype(np.int32)
    w = _workload(d, G, page, int(lens.max()), B=B, Hkv=Hkv, L=1, k=1)
    prob, sess, dp = H.setup(w, seed=41, seq_lens=[int(n) for n in lens])
    assert B * Hkv > torch.cuda.get_device_properties(0).multi_processor_count
    q_bits = prefill_queries(w, 23, B, pos.shape[1])
    got = H.to_f64(_run(sess, q_bits, pos, dp, 0))
    assert sess.read_status() == 0
    assert H.rel_err(got, _oracle(prob, q_bits, pos, 0)) <= H.TOL["bf16"]
    del sess, dp
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
