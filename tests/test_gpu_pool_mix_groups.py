"""The pool's bf16 mix with more than 16 channels and few tokens: the groups of 16
channels in CTAs of their own, or two or more of them in turn in one CTA where the
tokens nearly fill the SMs.  Every written key and value against the fp64 oracle."""
import pytest
import torch

from . import _harness as H
from .test_gpu_pool_mix import _w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,k,D,B", [
    (17, 17, 64, 1), (33, 33, 264, 2), (40, 40, 72, 130), (64, 49, 136, 60), (20, 18, 1096, 16), (32, 32, 64, 170)])
def test_channel_groups(L, k, D, B):
    prob, sess, dp = H.setup(_w(L, k, D, B, 2, Hkv=1), seed=13)
    sess.kv_mix(dp.h, dp.page_table, dp.slot)
    torch.cuda.synchronize()
    assert sess.read_status() == 0
    want = H.oracle_mix_tokens(prob)
    got = {bj: H.gpu_written_kv(sess, prob, *bj) for bj in want}
    for i in (0, 1):
        assert max(H.rel_err(got[bj][i], want[bj][i]) for bj in want) <= H.TOL["bf16"]
    del sess, dp
    torch.cuda.empty_cache()
