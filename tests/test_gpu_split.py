"""Frames that one block per multiprocessor covers: every pixel's atoms dealt over four threads (32 x 4 pixel tiles, eighty atoms
in flight), against the oracle at the edges of tiles, batches of atoms and forms."""
import numpy as np
import pytest
import torch

import oracle
import paper_2303_08999_b200 as sr
import sr_inputs
from gpu_util import dev, host, max_abs_err, signed_asymmetric_dictionary, signed_gamma, tol_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", ["f16", "f32"])
@pytest.mark.parametrize("n,c,h,w,r,D,k", [(1, 3, 2, 8, 4, 72, 5), (1, 3, 3, 11, 3, 12, 5), (2, 2, 5, 33, 1, 79, 3), (1, 4, 9, 16, 2, 80, 5), (1, 1, 4, 65, 1, 81, 7),
                                           (3, 3, 1, 1, 1, 161, 3), (1, 3, 64, 64, 2, 72, 5), (1, 3, 17, 31, 4, 33, 9), (1, 4, 6, 5, 3, 256, 9), (2, 1, 7, 43, 3, 40, 7)])
def test_dense(n, c, h, w, r, D, k, dt):
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("split", n, c, h, w, r, D=D, k=k, coef_dtype=dt))
    d = signed_asymmetric_dictionary(d, seed=k)
    args = (dev(lr), dev(coef), dev(d), r, k)
    want = oracle.dict_regress_dense(lr, coef, d, r, k)
    got = host(sr.sr_dict_regress_dense(*args))
    scale = max(1.0, np.abs(want).max())                      # (fp32 sums: errors grow with what is summed)
    assert max_abs_err(got, want) <= tol_for(coef) * scale
    clamped = np.clip(got, 0, 1)
    np.testing.assert_array_equal(host(sr.sr_dict_regress_dense(*args, sr.SR_CLAMP01)), clamped)
    np.testing.assert_array_equal(host(sr.sr_dict_regress_dense(*args, sr.SR_CLAMP01 | sr.SR_OUT_F16)), clamped.astype(np.float16))
    np.testing.assert_array_equal(host(sr.sr_dict_regress_dense(*args, sr.SR_OUT_U8)), np.rint(clamped * np.float32(255)).astype(np.uint8))


@pytest.mark.parametrize("dt", ["f16", "f32"])
@pytest.mark.parametrize("s,D,k,compact,gamma", [(12, 72, 5, False, True), (20, 96, 3, True, True), (81, 100, 5, False, False), (28, 28, 7, True, False)])
def test_subset(s, D, k, compact, gamma, dt):
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("split", 2, 3, 9, 21, 3, D=D, k=k, coef_dtype=dt))
    d = signed_asymmetric_dictionary(d, seed=k)
    idx = np.random.default_rng(s).permutation(D)[:s].astype(np.uint8)
    g = signed_gamma(s) if gamma else None
    flags, given = sr.SR_IDX_GLOBAL, coef
    if compact:
        flags, given = flags | sr.SR_COEF_COMPACT, np.ascontiguousarray(coef[:, idx])
    want = oracle.dict_regress_selected(lr, given, idx, g, d, 3, k, s, flags=flags)
    got = host(sr.sr_dict_regress_selected(dev(lr), dev(given), dev(idx), None if g is None else dev(g), dev(d), 3, k, s, flags))
    assert max_abs_err(got, want) <= tol_for(coef) * max(1.0, np.abs(want).max())


@pytest.mark.parametrize("dt", ["f16", "f32"])
def test_forced_general_kernel_is_the_thread_per_pixel_kernel(dt):
    # 5 blocks of 32 x 4 a frame: 30 frames are more than one block per multiprocessor takes, and too few for the row and the tiled kernel.
    # A pixel's sum is the same bits in either call; the split kernel's four parts have another order
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("split", 1, 3, 9, 9, 2, D=40, k=3, coef_dtype=dt))
    dlr, dco, ddi = dev(lr), dev(coef), dev(signed_asymmetric_dictionary(d, seed=3))
    by_rule = sr.sr_dict_regress_dense(dlr, dco, ddi, 2, 3)
    batch = sr.sr_dict_regress_dense(dlr.repeat(30, 1, 1, 1), dco.repeat(30, 1, 1, 1), ddi, 2, 3)
    sr.sr_test_force_kernel(0)
    try:
        forced = sr.sr_dict_regress_dense(dlr, dco, ddi, 2, 3)
    finally:
        sr.sr_test_force_kernel(-1)
    assert torch.equal(forced[0], batch[0]) and torch.equal(forced[0], batch[29])
    assert not torch.equal(forced, by_rule)


@pytest.mark.parametrize("c,D,k,split", [(4, 4, 7, False), (4, 5, 7, False), (4, 6, 7, True), (3, 12, 7, False), (3, 14, 7, True), (1, 25, 3, False), (1, 26, 3, True),
                                         (4, 2, 5, True), (3, 8, 5, True), (3, 7, 5, False)])
def test_few_atoms_and_channels_stay_with_the_thread_per_pixel_kernel(c, D, k, split):
    # the same bits as the pinned kernel's, or another order of the same sum
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("split", 1, c, 31, 33, 2, D=D, k=k, coef_dtype="f32"))
    args = (dev(lr), dev(coef), dev(signed_asymmetric_dictionary(d, seed=k)), 2, k)
    by_rule = sr.sr_dict_regress_dense(*args)
    sr.sr_test_force_kernel(0)
    try:
        forced = sr.sr_dict_regress_dense(*args)
    finally:
        sr.sr_test_force_kernel(-1)
    assert torch.equal(by_rule, forced) != split


@pytest.mark.parametrize("dt", ["f16", "f32"])
@pytest.mark.parametrize("k,D", [(3, 72), (5, 53), (9, 33)])
def test_coefficients_that_are_not_finite(k, D, dt):
    # in the first, the last and an inner atom: the same infinities and NaN as the sum has, in that pixel alone
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("split", 2, 3, 15, 33, 2, D=D, k=k, coef_dtype=dt))
    d = signed_asymmetric_dictionary(d, seed=k)
    d[D - 1] = np.abs(d[D - 1]) + 0.01                        # with finite taps of one sign: an infinity, not NaN
    clean = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), 2, k))
    bad, hit = coef.copy(), np.zeros(clean.shape, bool)
    for j, (f, y, x) in enumerate([(0, 0, 0), (0, 3, 31), (0, 4, 32), (1, 29, 65), (1, 28, 63), (0, 29, 64), (1, 13, 7), (1, 0, 65)]):
        bad[f, [D - 1, 0, D // 2][j % 3], y, x] = [np.inf, -np.inf, np.nan, np.inf][j % 4]
        hit[f, :, y, x] = True
    out = host(sr.sr_dict_regress_dense(dev(lr), dev(bad), dev(d), 2, k))
    np.testing.assert_array_equal(out[~hit], clean[~hit])
    want = oracle.dict_regress_dense(lr, bad, d, 2, k)[hit]
    np.testing.assert_array_equal(np.isnan(out[hit]), np.isnan(want))
    np.testing.assert_array_equal(out[hit][~np.isnan(want)], want[~np.isnan(want)].astype(np.float32))
    assert np.isinf(want).any() and np.isnan(want).any()
