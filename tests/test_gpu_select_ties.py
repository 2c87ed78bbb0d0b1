"""Ties at the threshold of the selection made inside the tensor-core regression: the same choice as the oracle's whatever share of
the pixels has them, in a time that does not depend on it."""
import numpy as np
import pytest
import torch

import oracle
import paper_2303_08999_b200 as sr
from gpu_util import dev, host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,s", [(9, 8), (16, 1), (33, 7), (40, 8), (72, 8), (72, 4), (72, 16), (97, 9), (128, 8), (8, 8)])
@pytest.mark.parametrize("share", [0.0, 0.01, 0.13, 1.0])
def test_ties_at_the_threshold(D, s, share):
    rng = np.random.default_rng(1000 * D + 10 * s + int(100 * share))
    H, W = 24, 136
    rank = np.argsort(rng.random((D, H, W)), axis=0)                          # rank of every atom, 0 the largest
    mag = 0.75 - np.arange(D) * 2.0 ** -9                                     # exact in binary16, all different
    per_rank = np.broadcast_to(mag[:, None, None], (D, H, W)).copy()
    for y, x in np.argwhere(rng.random((H, W)) < share):
        lo, hi = s - 1 - rng.integers(0, min(3, s)), min(D - 1, s - 1 + rng.integers(1, 40))
        per_rank[lo:hi + 1, y, x] = per_rank[lo, y, x]                        # ranks lo .. hi tie, the threshold among them
    for y, x in np.argwhere(rng.random((H, W)) < 0.05):
        per_rank[rng.integers(0, s + 1):, y, x] = 0.0                         # fewer than s that are not zero
    coef = np.take_along_axis(per_rank, rank, axis=0) * rng.choice([-1, 1], (D, H, W))
    coef = np.ascontiguousarray(coef[None].astype(np.float16))
    # an atom that reads the centre alone, scaled by its index, tells the choice
    d = np.zeros((D, 9), np.float32)
    d[:, 4] = 1.0 + np.arange(D) / 8.0
    idx, sel = oracle.dict_select(coef, s, want_sel=True)
    want = (sel * d[idx, 4]).sum(1)[:, None]
    got = host(sr.sr_dict_regress_selected(dev(np.ones((1, 1, H, W), np.float32)), dev(coef), None, None, dev(d), 1, 3, s))
    # exact products of at most 0.75 x 16.9, s sums of at most 12.7 s rounded (or cut off) to 24 bits; another choice differs by 0.03
    assert np.abs(got - want).max() <= 2.0 ** -23 * 12.7 * s * (s + 2)
    assert sr.sr_device_status() == 0


def test_ties_at_the_largest_magnitude():
    # the threshold's next magnitude is infinity there
    D, s, H, W = 40, 8, 16, 128
    rng = np.random.default_rng(5)
    coef = (rng.integers(0, 3, (1, D, H, W)) * 32752.0 * rng.choice([-1, 1], (1, D, H, W))).astype(np.float16)
    assert np.abs(coef.astype(np.float32)).max() == 65504
    d = np.zeros((D, 9), np.float32)
    d[:, 4] = 1.0 + np.arange(D) / 8.0
    idx, sel = oracle.dict_select(coef, s, want_sel=True)
    want = (sel * d[idx, 4]).sum(1)[:, None]
    got = host(sr.sr_dict_regress_selected(dev(np.ones((1, 1, H, W), np.float32)), dev(coef), None, None, dev(d), 1, 3, s))
    assert np.abs(got - want).max() <= 2.0 ** -23 * 65504 * 6 * s * (s + 2)
    assert sr.sr_device_status() == 0


def _device_us(call, reps):
    call()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(reps):
            call()
    times = []
    for _ in range(9):
        first, last = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        first.record()
        graph.replay()
        last.record()
        torch.cuda.synchronize()
        times.append(first.elapsed_time(last) * 1e3 / reps)
    return sorted(times)[4]


@pytest.mark.parametrize("s,D", [(4, 72), (8, 72), (16, 128)])
def test_time_does_not_depend_on_ties(s, D):
    # one pixel in a hundred with ties, every pixel with them, and rows of either kind in turn (1.4 to 1.5 times as long where tied
    # pixels were work of their own)
    g = torch.Generator(device="cuda").manual_seed(1)
    lr, d = torch.rand(1, 3, 135, 240, generator=g, device="cuda"), torch.rand(D, 25, generator=g, device="cuda")
    few = (torch.randn(1, D, 540, 960, generator=g, device="cuda") * 0.05 + 1.0 / D).half()
    flat = torch.full_like(few, 0.25)
    turns = torch.where((torch.arange(540, device="cuda") % 2 == 0).view(1, 1, -1, 1), few, flat)
    out = torch.empty(1, 3, 540, 960, device="cuda")
    us = [_device_us(lambda c=c: sr.sr_dict_regress_selected(lr, c, None, None, d, 4, 5, s, 0, out=out), 20) for c in (few, flat, turns)]
    assert max(us) <= 1.15 * us[0]
