"""Calls of different contexts beside each other on one GPU: each gives what it gives alone, whatever share of the SMs it finds.

A prefill's CTAs wait for one another's tiles, but only for tiles that a running CTA has taken, so a launch of which a part has
no room yet still ends.  Beside it may run what ends by itself or waits for SMs that the prefill gives back: a decode step (a CTA
per SM that wait for one another), another prefill.  One decode stream only: two of them could each hold SMs that the other needs.
"""
import pytest
import torch

from synth import workloads as W
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


def shape(d, f, E=8, k=2, r=0):
    return W.LayerShape("t", 9, d, f, n_experts=E, top_k=k, wd_rank=r)


@pytest.mark.parametrize("beside", [
    (shape(1024, 2816), 1, 40),                         # decode, dense experts
    (shape(1024, 2816), 8, 20),
    (shape(1024, 1024, r=128), 1, 40),                  # decode, decomposed experts
    (shape(512, 1536, E=16), 600, 12),                  # another prefill
    (shape(512, 1024, r=64), 600, 12),
], ids=["decode-T1", "decode-T8", "wd-decode-T1", "prefill", "wd-prefill"])
@pytest.mark.parametrize("first", ["prefill in front", "prefill behind"])
def test_prefill_beside_another_contexts_calls(beside, first):
    sh2, T2, n2 = beside
    lay1, t1, _ = U.build(shape(1024, 2816), 700)
    lay2, t2, _ = U.build(sh2, T2)
    x1 = [t1["x"], t1["x"].flip(0).contiguous()]
    x2 = [t2["x"], t2["x"].roll(1, -1).contiguous()]
    want1, want2 = [lay1.forward(x) for x in x1], [lay2.forward(x) for x in x2]
    torch.cuda.synchronize()
    low, high = torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-1)
    s1, s2 = (high, low) if first == "prefill in front" else (low, high)
    got1, got2 = [], []
    n1 = 10
    for i in range(max(n1, n2)):                        # enqueued faster than they run: the streams stay busy together
        if i < n1:
            with torch.cuda.stream(s1):
                got1.append(lay1.forward(x1[i & 1]))
        if i < n2:
            with torch.cuda.stream(s2):
                got2.append(lay2.forward(x2[i & 1]))
    torch.cuda.synchronize()
    assert lay1.check() == 0 and lay2.check() == 0
    for i, y in enumerate(got1):
        assert torch.equal(y, want1[i & 1]), f"prefill {i}"
    for i, y in enumerate(got2):
        assert torch.equal(y, want2[i & 1]), f"the other context's call {i}"
