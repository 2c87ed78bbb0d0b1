"""Ties at the threshold of the selection made inside the tensor-core regression: a chunk of 64 pixels takes its pixels with
too many coefficients one by one while there are up to eight, and all of its atoms in one pass beyond that."""
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
