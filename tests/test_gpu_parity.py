"""Parity of the CUDA library (called through its C ABI) against the fp64 CPU oracle.

Small cases are compared element by element; they span several tiles, ragged tails, every atom size
and both coefficient types. Index outputs must be bit-exact; pixel values within 1e-5 (fp32
coefficients) or 2e-3 (binary16 coefficients) max abs error.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2303_08999_b200 as sr
import sr_inputs
from gpu_util import TOL_F16, TOL_F32, dev, host, max_abs_err, on_kernel, signed_asymmetric_dictionary, signed_gamma, tol_for

pytestmark = pytest.mark.gpu


def _wl(n, c, h, w, r, D, k, dt):
    return sr_inputs.Workload("t", n, c, h, w, r, D=D, k=k, coef_dtype=dt)


# ------------------------------------------------------------------ stage 1

@pytest.mark.parametrize("n,c,h,w,r", [(1, 3, 64, 64, 2), (2, 3, 37, 53, 3), (1, 1, 5, 300, 4), (1, 2, 1, 1, 2),
                                       (1, 3, 9, 7, 1), (1, 1, 6, 5, 8), (1, 4, 2, 3, 5), (1, 3, 41, 35, 3), (2, 1, 9, 11, 6),
                                       (1, 2, 13, 10, 5), (1, 1, 7, 9, 7)])
def test_bicubic(n, c, h, w, r):
    lr = sr_inputs.make_lr(_wl(n, c, h, w, r, 1, 1, "f32"))
    got = host(sr.sr_bicubic_upsample(dev(lr), r))
    want = oracle.bicubic_upsample(lr, r)
    assert max_abs_err(got, want) <= 1e-6


@pytest.mark.parametrize("n,c,h,w,r", [(2, 1, 720, 700, 3), (1, 3, 251, 401, 3), (1, 3, 271, 481, 4), (1, 2, 511, 515, 2),
                                       (300, 3, 9, 7, 3), (70, 2, 32, 32, 2), (40, 1, 2000, 1, 1), (3, 3, 700, 5, 2), (33, 3, 5, 2, 8)])
def test_bicubic_runs_of_blocks(n, c, h, w, r):          # a thread walks several blocks; the last run is cut short
    test_bicubic(n, c, h, w, r)


# ------------------------------------------------------------------ dense

DENSE_CASES = [
    # n, c, h, w, r, D, k, dtype
    (1, 3, 64, 64, 2, 72, 5, "f32"),      # cfg0 in full
    (1, 3, 64, 64, 2, 72, 5, "f16"),
    (2, 3, 33, 50, 4, 72, 5, "f16"),      # ragged in both directions, two frames
    (1, 3, 20, 67, 3, 72, 5, "f16"),
    (1, 1, 40, 24, 2, 16, 3, "f16"),
    (1, 3, 24, 40, 2, 32, 7, "f16"),
    (1, 3, 12, 40, 4, 128, 5, "f16"),
    (1, 3, 10, 24, 2, 256, 3, "f16"),
    (1, 5, 9, 16, 2, 7, 9, "f32"),        # odd atom count, five channels, largest atom
    (1, 3, 7, 5, 3, 3, 1, "f32"),         # 1x1 atoms
    (1, 3, 1, 1, 2, 72, 5, "f16"),        # a single LR pixel
    (1, 3, 3, 100, 4, 72, 5, "f16"),      # HR width 400: not a multiple of 128
    (1, 3, 30, 35, 4, 72, 5, "f16"),      # HR width 140: not a multiple of 8
]


# The host rules (-1) give most of these frames to the split kernel; the kernels they were written for, the general one, both
# layouts and the subset and gather kernels, stay tested by pinning each in turn (where it does not take a call, the rules do).
ON_KERNELS = pytest.mark.parametrize("kernel", [-1, 0, 1, 2, 3, 4])


@pytest.mark.parametrize("case", DENSE_CASES, ids=lambda c: "-".join(map(str, c)))
@pytest.mark.parametrize("clamp", [0, 1])
@pytest.mark.parametrize("kernel", [-1, 0, 1, 2])
def test_dense(case, clamp, kernel):
    n, c, h, w, r, D, k, dt = case
    lr, dict_, coef = sr_inputs.make_inputs(_wl(n, c, h, w, r, D, k, dt))
    if k == 1:  # a difference of Gaussians has no 1x1 form (0/0): use plain seeded weights instead
        dict_ = np.random.default_rng(1).uniform(-1, 1, dict_.shape).astype(np.float32)
    flags = sr.SR_CLAMP01 if clamp else 0
    with on_kernel(kernel):
        got = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(dict_), r, k, flags))
    want = oracle.dict_regress_dense(lr, coef, dict_, r, k, flags=flags)
    assert sr.sr_device_status() == 0
    assert max_abs_err(got, want) <= tol_for(coef)


@pytest.mark.parametrize("kernel", [1, 2])                   # first, second tensor-core layout
@pytest.mark.parametrize("case", [(1, 3, 24, 40, 2, 16, 3), (2, 1, 33, 48, 2, 8, 5), (1, 2, 20, 72, 3, 17, 5), (1, 3, 24, 40, 2, 32, 7), (1, 3, 20, 32, 1, 16, 1),
                                  (2, 3, 9, 34, 4, 1, 5), (1, 1, 40, 56, 1, 33, 3), (1, 2, 17, 40, 4, 24, 7)], ids=lambda c: "-".join(map(str, c)))
def test_both_layouts_on_small_frames_of_few_atoms(kernel, case):
    # the host rules give such frames to the split and the general kernel; what the layouts do with them stays tested
    n, c, h, w, r, D, k = case
    lr, d, coef = sr_inputs.make_inputs(_wl(n, c, h, w, r, D, k, "f16"))
    d = signed_asymmetric_dictionary(d, seed=k) if k > 1 else np.random.default_rng(1).uniform(-1, 1, d.shape).astype(np.float32)
    s = min(D, 12)
    S, gamma = np.arange(D - 1, D - 1 - s, -1).astype(np.uint8), signed_gamma(s)
    sr.sr_test_force_kernel(kernel)
    try:
        dense = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), r, k))
        subset = host(sr.sr_dict_regress_selected(dev(lr), dev(coef), dev(S), dev(gamma), dev(d), r, k, s, sr.SR_IDX_GLOBAL))
    finally:
        sr.sr_test_force_kernel(-1)
    assert sr.sr_device_status() == 0
    assert max_abs_err(dense, oracle.dict_regress_dense(lr, coef, d, r, k)) <= TOL_F16
    assert max_abs_err(subset, oracle.dict_regress_selected(lr, coef, S, gamma, d, r, k, s, flags=oracle.IDX_GLOBAL)) <= TOL_F16


def test_dense_is_deterministic_and_leaves_inputs_alone():
    lr, dict_, coef = sr_inputs.make_inputs(_wl(2, 3, 33, 50, 4, 72, 5, "f16"))
    dlr, dco, ddi = dev(lr), dev(coef), dev(dict_)
    a = host(sr.sr_dict_regress_dense(dlr, dco, ddi, 4, 5))
    b = host(sr.sr_dict_regress_dense(dlr, dco, ddi, 4, 5))
    np.testing.assert_array_equal(a, b)
    np.testing.assert_array_equal(host(dco), coef)
    np.testing.assert_array_equal(host(dlr), lr)


def test_dense_delta_atom_reproduces_bicubic_on_gpu():
    wl = _wl(1, 3, 20, 48, 4, 72, 5, "f16")
    lr, dict_, _ = sr_inputs.make_inputs(wl)
    dict_[0] = 0
    dict_[0, 12] = 1
    coef = np.zeros((1, 72, wl.H, wl.W), np.float16)
    coef[:, 0] = 1
    got = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(dict_), 4, 5))
    up = host(sr.sr_bicubic_upsample(dev(lr), 4))
    assert max_abs_err(got, up.astype(np.float64)) <= 1e-6
    assert max_abs_err(got, oracle.bicubic_upsample(lr, 4)) <= 1e-6


def test_dense_on_a_side_stream_and_offset_views():
    """Pointers that are element-aligned but not 16-byte aligned still work (general path)."""
    wl = _wl(1, 3, 16, 24, 2, 16, 3, "f16")
    lr, dict_, coef = sr_inputs.make_inputs(wl)
    buf = torch.empty(coef.size + 1, dtype=torch.float16, device="cuda")
    view = buf[1:].view(coef.shape)
    view.copy_(dev(coef))
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(st):
        got = sr.sr_dict_regress_dense(dev(lr), view, dev(dict_), 2, 3)
    st.synchronize()
    assert max_abs_err(host(got), oracle.dict_regress_dense(lr, coef, dict_, 2, 3)) <= TOL_F16


# ------------------------------------------------------------------ selection

def _coarse(coef):
    """Quantise to a coarse grid so that exact magnitude ties, +/- pairs and zeros are frequent."""
    return (np.round(coef.astype(np.float32) * 64) / 64).astype(coef.dtype)


@pytest.mark.parametrize("dt", ["f16", "f32"])
@pytest.mark.parametrize("D,s", [(72, 8), (72, 1), (72, 4), (72, 16), (72, 20), (72, 72), (16, 16), (128, 8), (256, 5), (5, 3)])
def test_select_bit_exact(dt, D, s):
    wl = _wl(2, 1, 9, 23, 2, D, 1, dt)
    for coef in (sr_inputs.make_coef(wl), _coarse(sr_inputs.make_coef(wl, seed=5))):
        idx, sel = sr.sr_dict_select(dev(coef), s, want_sel=True)
        want_idx, want_sel = oracle.dict_select(coef, s, want_sel=True)
        np.testing.assert_array_equal(host(idx), want_idx)
        np.testing.assert_array_equal(host(sel).astype(np.float64), want_sel)
        np.testing.assert_array_equal(host(sr.sr_dict_select(dev(coef), s)), want_idx)


@pytest.mark.parametrize("dt", ["f16", "f32"])
@pytest.mark.parametrize("n,h,w", [(1, 9, 23), (2, 5, 6), (1, 1, 1), (2, 2, 27)])
@pytest.mark.parametrize("D,s", [(1, 1), (2, 2), (7, 4), (8, 4), (9, 5), (16, 8), (17, 9), (64, 8), (65, 16), (128, 15), (129, 8), (256, 16)])
def test_select_any_width_with_magnitudes_that_differ_in_few_bits(dt, n, h, w, D, s):
    rng = np.random.default_rng(D * 31 + s)
    top = (n, D, h, w)
    bits = rng.integers(0, 3, top) * 5 + rng.integers(0, 130, top) * (rng.random(top) < 0.5)      # exact ties and neighbours
    base, kind = (np.float32(0.5).view(np.uint32), np.uint32) if dt == "f32" else (np.float16(0.5).view(np.uint16), np.uint16)
    coef = (base + bits.astype(kind)).astype(kind).view(np.float32 if dt == "f32" else np.float16)
    coef = coef * rng.choice([-1, 1], top).astype(coef.dtype) * (rng.random(top) < 0.8)           # signs, and some zeros
    coef = np.ascontiguousarray(coef.astype(np.float32 if dt == "f32" else np.float16))
    idx, sel = sr.sr_dict_select(dev(coef), s, want_sel=True)
    want_idx, want_sel = oracle.dict_select(coef, s, want_sel=True)
    np.testing.assert_array_equal(host(idx), want_idx)
    np.testing.assert_array_equal(host(sel).astype(np.float64), want_sel)
    # the selection made inside the regression: an atom that reads the centre alone, scaled by its index, tells the choice
    lr, d = np.ones((n, 1, h, w), np.float32), np.zeros((D, 9), np.float32)
    d[:, 4] = 1.0 + np.arange(D) / 8.0
    got = host(sr.sr_dict_regress_selected(dev(lr), dev(coef), None, None, dev(d), 1, 3, s))
    want = (want_sel * d[want_idx, 4]).sum(1)[:, None]
    # s products of at most 0.53 x 33, summed in fp32
    assert np.abs(got - want).max() <= 2.0 ** -23 * s * s * 18


@pytest.mark.parametrize("kind", ["widened", "rectified", "one tiny value"])
@pytest.mark.parametrize("D,s", [(1, 1), (3, 1), (9, 1), (72, 1), (8, 2), (130, 2), (72, 3), (72, 8), (200, 16), (256, 17)])
def test_fp32_selection_where_magnitudes_repeat(kind, D, s):
    # repeated magnitudes whose dropped bits are all zero need no second look; one coefficient with such bits brings it back
    rng = np.random.default_rng(D + s)
    coef = rng.integers(-3, 4, (2, D, 7, 23)).astype(np.float16).astype(np.float32) * np.float32(0.125)
    if kind == "rectified":
        coef = np.maximum(rng.standard_normal(coef.shape), 0).astype(np.float32) * (rng.random(coef.shape) < 0.3)
    elif kind == "one tiny value":                            # a magnitude below the key's lowest bit, behind equal zeros
        coef[:, D - 1] = np.where(rng.random((2, 7, 23)) < 0.5, np.float32(1e-44), np.nextafter(np.float32(0.375), np.float32(1)))
    coef = np.ascontiguousarray(coef.astype(np.float32))
    idx, sel = sr.sr_dict_select(dev(coef), s, want_sel=True)
    want_idx, want_sel = oracle.dict_select(coef, s, want_sel=True)
    np.testing.assert_array_equal(host(idx), want_idx)
    np.testing.assert_array_equal(host(sel).astype(np.float64), want_sel)
    lr, d = np.ones((2, 1, 7, 23), np.float32), np.zeros((D, 9), np.float32)
    d[:, 4] = 1.0 + np.arange(D) / 8.0
    got = host(sr.sr_dict_regress_selected(dev(lr), dev(coef), None, None, dev(d), 1, 3, s))
    want = (want_sel * d[want_idx, 4]).sum(1)[:, None]
    # s products of at most 4 x 33, summed in fp32
    assert np.abs(got - want).max() <= 2.0 ** -23 * s * s * 132


def test_select_signed_zero_and_extremes():
    coef = np.zeros((1, 8, 2, 8), np.float16)
    coef[0, 3] = -0.0
    coef[0, 5, 0, :] = [65504, -65504, 6e-8, -6e-8, 1, -1, 0.5, 0]
    coef[0, 6, 0, :] = [-65504, 65504, -6e-8, 6e-8, -1, 1, 0.25, -0.0]
    np.testing.assert_array_equal(host(sr.sr_dict_select(dev(coef), 3)), oracle.dict_select(coef, 3))


# ------------------------------------------------------------------ selected regression

SEL_CASES = [
    (1, 3, 33, 50, 4, 72, 5, "f16", 8),
    (2, 3, 20, 30, 2, 72, 5, "f32", 8),
    (1, 3, 16, 40, 3, 32, 3, "f16", 4),
    (1, 1, 12, 24, 2, 128, 7, "f16", 16),
    (1, 3, 8, 24, 2, 72, 5, "f16", 20),
    (1, 3, 8, 24, 2, 16, 5, "f16", 16),
    # widths that are multiples of 16: the index-listed and compact modes take the tensor-core kernel too
    (1, 3, 24, 64, 2, 72, 5, "f16", 8),
    (1, 3, 20, 36, 4, 32, 3, "f16", 4),
    (2, 3, 9, 40, 2, 128, 5, "f16", 8),
    (1, 3, 10, 24, 2, 20, 5, "f16", 3),
    (1, 2, 40, 72, 4, 72, 3, "f16", 8),
    (1, 3, 7, 168, 2, 6, 7, "f16", 6),
    # 8 < s <= 16: the sixteen-entry list of the in-kernel selection, two rank halves per lane in the listed modes
    (1, 3, 12, 32, 2, 72, 5, "f16", 12),
    (1, 3, 12, 64, 4, 128, 3, "f16", 16),
    (1, 3, 10, 40, 2, 24, 5, "f16", 9),
]


@pytest.mark.parametrize("case", SEL_CASES, ids=lambda c: "-".join(map(str, c)))
@ON_KERNELS
def test_selected_all_modes(case, kernel):
    with on_kernel(kernel):
        _selected_all_modes(case)


def _selected_all_modes(case):
    n, c, h, w, r, D, k, dt, s = case
    wl = _wl(n, c, h, w, r, D, k, dt)
    lr, dict_, coef = sr_inputs.make_inputs(wl)
    tol = tol_for(coef)
    dlr, dco, ddi = dev(lr), dev(coef), dev(dict_)
    want = oracle.dict_regress_selected(lr, coef, None, None, dict_, r, k, s, flags=oracle.CLAMP01)
    # top-s chosen inside the call
    got = host(sr.sr_dict_regress_selected(dlr, dco, None, None, ddi, r, k, s, sr.SR_CLAMP01))
    assert max_abs_err(got, want) <= tol
    # two-step: select, then regress from the index planes (full tensor, then compact values)
    idx, sel = sr.sr_dict_select(dco, s, want_sel=True)
    got = host(sr.sr_dict_regress_selected(dlr, dco, idx, None, ddi, r, k, s, sr.SR_CLAMP01))
    assert max_abs_err(got, want) <= tol
    got = host(sr.sr_dict_regress_selected(dlr, sel, idx, None, ddi, r, k, s, sr.SR_CLAMP01 | sr.SR_COEF_COMPACT))
    assert max_abs_err(got, want) <= tol
    # the paper's global subset with re-weights
    rng = np.random.default_rng(3)
    S = rng.choice(D, size=s, replace=False).astype(np.uint8)
    gamma = rng.uniform(0.5, 1.5, size=s).astype(np.float32)
    want = oracle.dict_regress_selected(lr, coef, S, gamma, dict_, r, k, s, flags=oracle.IDX_GLOBAL)
    got = host(sr.sr_dict_regress_selected(dlr, dco, dev(S), dev(gamma), ddi, r, k, s, sr.SR_IDX_GLOBAL))
    assert max_abs_err(got, want) <= tol
    compact = dev(coef[:, S.astype(int)].copy())
    got = host(sr.sr_dict_regress_selected(dlr, compact, dev(S), dev(gamma), ddi, r, k, s,
                                           sr.SR_IDX_GLOBAL | sr.SR_COEF_COMPACT))
    assert max_abs_err(got, want) <= tol
    want = oracle.dict_regress_selected(lr, coef, S, None, dict_, r, k, s, flags=oracle.IDX_GLOBAL)
    got = host(sr.sr_dict_regress_selected(dlr, dco, dev(S), None, ddi, r, k, s, sr.SR_IDX_GLOBAL))
    assert max_abs_err(got, want) <= tol
    assert sr.sr_device_status() == 0


def test_selected_with_s_equal_D_is_dense():
    wl = _wl(1, 3, 16, 24, 2, 16, 5, "f16")
    lr, dict_, coef = sr_inputs.make_inputs(wl)
    a = host(sr.sr_dict_regress_selected(dev(lr), dev(coef), None, None, dev(dict_), 2, 5, 16))
    assert max_abs_err(a, oracle.dict_regress_dense(lr, coef, dict_, 2, 5)) <= TOL_F16


@pytest.mark.parametrize("D,s,w", [(72, 8, 24), (128, 5, 64), (24, 8, 32), (72, 1, 24), (72, 13, 32), (40, 16, 24)])
def test_selected_with_ties(D, s, w):
    wl = _wl(1, 3, 16, w, 2, D, 5, "f16")
    lr, dict_, coef = sr_inputs.make_inputs(wl)
    coef = _coarse(coef)
    want = oracle.dict_regress_selected(lr, coef, None, None, dict_, 2, 5, s)
    got = host(sr.sr_dict_regress_selected(dev(lr), dev(coef), None, None, dev(dict_), 2, 5, s))
    assert max_abs_err(got, want) <= TOL_F16
    # the same pixels through explicit index planes (ties resolved by sr_dict_select) and compact values
    idx, sel = sr.sr_dict_select(dev(coef), s, want_sel=True)
    np.testing.assert_array_equal(host(idx), oracle.dict_select(coef, s))
    got = host(sr.sr_dict_regress_selected(dev(lr), dev(coef), idx, None, dev(dict_), 2, 5, s))
    assert max_abs_err(got, want) <= TOL_F16
    got = host(sr.sr_dict_regress_selected(dev(lr), sel, idx, None, dev(dict_), 2, 5, s, sr.SR_COEF_COMPACT))
    assert max_abs_err(got, want) <= TOL_F16


# Frames whose tile counts lie on both sides of the tile-height and layout rules: 8-row tiles in one, two and three turns of
# the SMs, 16-row tiles, the row kernel and the general kernel for few atoms and short lists.
@pytest.mark.parametrize("n,h,w,r,D,k,s", [(1, 272, 320, 2, 20, 3, 4), (1, 150, 200, 2, 40, 5, 8), (2, 64, 64, 2, 16, 5, 16), (1, 31, 48, 4, 16, 3, 3),
                                           (3, 37, 56, 2, 32, 7, 4), (1, 65, 112, 3, 128, 3, 8), (1, 117, 160, 3, 16, 5, 5)])
def test_layout_rules_of_small_and_middling_frames(n, h, w, r, D, k, s):
    wl = _wl(n, 1, h, w, r, D, k, "f16")
    lr, d, coef = sr_inputs.make_inputs(wl)
    d = signed_asymmetric_dictionary(d, seed=k)
    want = oracle.dict_regress_dense(lr, coef, d, r, k)
    assert max_abs_err(host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), r, k)), want) <= TOL_F16
    want = oracle.dict_regress_selected(lr, coef, None, None, d, r, k, s)
    assert max_abs_err(host(sr.sr_dict_regress_selected(dev(lr), dev(coef), None, None, dev(d), r, k, s)), want) <= TOL_F16
    idx, sel = sr.sr_dict_select(dev(coef), s, want_sel=True)
    got = host(sr.sr_dict_regress_selected(dev(lr), sel, idx, None, dev(d), r, k, s, sr.SR_COEF_COMPACT))
    assert max_abs_err(got, want) <= TOL_F16
    assert sr.sr_device_status() == 0


# ------------------------------------------------------------------ orientation and sign of the taps

SIGNED_CASES = [
    # n, c, h, w, r, D, k, dtype, s
    (1, 3, 24, 64, 2, 72, 5, "f16", 8),    # the tensor-core kernel takes every mode
    (2, 3, 33, 50, 4, 72, 5, "f16", 8),    # HR width 200: dense / in-kernel selection / subset on the tensor cores, index planes on the general kernel
    (1, 3, 20, 30, 2, 72, 5, "f32", 8),    # fp32 coefficients: general and split kernel
    (1, 3, 12, 40, 2, 32, 7, "f16", 4),
    (1, 3, 12, 32, 2, 72, 3, "f16", 12),
    (1, 1, 9, 16, 2, 7, 9, "f32", 3),      # 9 x 9 atoms: general kernel
    (1, 3, 30, 35, 4, 72, 5, "f16", 8),    # HR width 140: general and split kernel with binary16 coefficients
    (1, 3, 40, 64, 4, 72, 5, "f16", 8),    # several 16-row tiles, two tile columns
]


@pytest.mark.parametrize("case", SIGNED_CASES, ids=lambda c: "-".join(map(str, c)))
@ON_KERNELS
def test_signed_asymmetric_dictionary_and_negative_gamma_all_modes(case, kernel):
    with on_kernel(kernel):
        _signed_all_modes(case)


def _signed_all_modes(case):
    """Atoms without any symmetry and with both signs, re-weights with both signs: a 180-degree tap flip, a transposed
    patch or a lost sign in the binary16 hi / lo split of the dictionary fails here (it passes with the generator's
    point-symmetric, non-negative atoms)."""
    n, c, h, w, r, D, k, dt, s = case
    wl = _wl(n, c, h, w, r, D, k, dt)
    lr, dict_, coef = sr_inputs.make_inputs(wl)
    dict_ = signed_asymmetric_dictionary(dict_)
    assert (dict_ < 0).any() and not np.allclose(dict_.reshape(D, k, k), dict_.reshape(D, k, k)[:, ::-1, ::-1])
    tol = tol_for(coef)
    dlr, dco, ddi = dev(lr), dev(coef), dev(dict_)
    got = host(sr.sr_dict_regress_dense(dlr, dco, ddi, r, k))
    assert max_abs_err(got, oracle.dict_regress_dense(lr, coef, dict_, r, k)) <= tol
    want = oracle.dict_regress_selected(lr, coef, None, None, dict_, r, k, s)
    got = host(sr.sr_dict_regress_selected(dlr, dco, None, None, ddi, r, k, s))
    assert max_abs_err(got, want) <= tol
    idx, sel = sr.sr_dict_select(dco, s, want_sel=True)
    got = host(sr.sr_dict_regress_selected(dlr, dco, idx, None, ddi, r, k, s))
    assert max_abs_err(got, want) <= tol
    got = host(sr.sr_dict_regress_selected(dlr, sel, idx, None, ddi, r, k, s, sr.SR_COEF_COMPACT))
    assert max_abs_err(got, want) <= tol
    rng = np.random.default_rng(5)
    S = rng.choice(D, size=s, replace=False).astype(np.uint8)
    S[0] = 1 if 1 not in S[1:] else S[0]                     # the off-centre delta atom is in the subset
    gamma = signed_gamma(s)
    assert (gamma < 0).any()
    want = oracle.dict_regress_selected(lr, coef, S, gamma, dict_, r, k, s, flags=oracle.IDX_GLOBAL)
    got = host(sr.sr_dict_regress_selected(dlr, dco, dev(S), dev(gamma), ddi, r, k, s, sr.SR_IDX_GLOBAL))
    assert max_abs_err(got, want) <= tol
    compact = dev(coef[:, S.astype(int)].copy())
    got = host(sr.sr_dict_regress_selected(dlr, compact, dev(S), dev(gamma), ddi, r, k, s, sr.SR_IDX_GLOBAL | sr.SR_COEF_COMPACT))
    assert max_abs_err(got, want) <= tol
    assert sr.sr_device_status() == 0


@pytest.mark.parametrize("dt,w", [("f16", 48), ("f32", 48), ("f16", 35)])
@pytest.mark.parametrize("tap", [(0, 1), (4, 0), (3, 4), (2, 2)])
@ON_KERNELS
def test_off_centre_delta_atom_shifts_the_upsampled_image(dt, w, tap, kernel):
    with on_kernel(kernel):
        _off_centre_delta(dt, w, tap)


def _off_centre_delta(dt, w, tap):
    """One atom that is a single tap at (a, b), one-hot coefficients: the output is the up-sampled image read at
    (Y + a - p, X + b - p), clamped to the frame. The expected frame is built from the bicubic oracle by indexing
    alone, so the pairing of taps and patch positions is checked without the oracle's own regression."""
    a, b = tap
    r, k, D, p = 4, 5, 72, 2
    wl = _wl(1, 3, 20, w, r, D, k, dt)
    lr, dict_, _ = sr_inputs.make_inputs(wl)
    dict_[3] = 0
    dict_[3, a * k + b] = 1
    coef = np.zeros((1, D, wl.H, wl.W), np.float16 if dt == "f16" else np.float32)
    coef[:, 3] = 1
    U = oracle.bicubic_upsample(lr, r)
    yy = np.clip(np.arange(wl.H) + a - p, 0, wl.H - 1)
    xx = np.clip(np.arange(wl.W) + b - p, 0, wl.W - 1)
    want = U[:, :, yy][:, :, :, xx]
    dlr, dco, ddi = dev(lr), dev(coef), dev(dict_)
    assert max_abs_err(host(sr.sr_dict_regress_dense(dlr, dco, ddi, r, k)), want) <= 2e-6
    assert max_abs_err(host(sr.sr_dict_regress_selected(dlr, dco, None, None, ddi, r, k, 3)), want) <= 2e-6
    S = np.array([0, 3, 5], np.uint8)
    assert max_abs_err(host(sr.sr_dict_regress_selected(dlr, dco, dev(S), None, ddi, r, k, 3, sr.SR_IDX_GLOBAL)), want) <= 2e-6
    idx, sel = sr.sr_dict_select(dco, 3, want_sel=True)
    assert max_abs_err(host(sr.sr_dict_regress_selected(dlr, sel, idx, None, ddi, r, k, 3, sr.SR_COEF_COMPACT)), want) <= 2e-6
    np.testing.assert_allclose(oracle.dict_regress_dense(lr, coef, dict_, r, k), want, rtol=0, atol=1e-12)


@pytest.mark.parametrize("scale,bound", [(2.0 ** 15, TOL_F16 * 2.0 ** 15), (2.0 ** -10, 1e-5)])
@pytest.mark.parametrize("kernel", [-1, 1, 2])
def test_dictionary_magnitude_range_of_the_tensor_core_path(scale, bound, kernel):
    with on_kernel(kernel):
        _dictionary_magnitude_range(scale, bound)


def _dictionary_magnitude_range(scale, bound):
    """The tensor-core path keeps the fp32 dictionary as a binary16 hi + lo pair, so its taps must stay below the
    largest binary16 number (65504); taps below 2^-14 fall into the binary16 subnormals and keep an absolute, not a
    relative, precision (2^-25 per tap). A large dictionary (taps up to about 9500) must be as accurate relative to
    its scale as the ordinary one; a tiny one (taps around 1e-4) within the absolute bound that follows from 2^-25 per
    tap: 3 (sum of |coefficients|) x 25 taps x 1.45 (|U|) x 2^-25 = 3.3e-6."""
    wl = _wl(1, 3, 24, 64, 2, 72, 5, "f16")
    lr, dict_, coef = sr_inputs.make_inputs(wl)
    dict_ = (signed_asymmetric_dictionary(dict_) * np.float32(scale)).astype(np.float32)
    assert np.abs(dict_).max() < 65504
    got = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(dict_), 2, 5))
    assert max_abs_err(got, oracle.dict_regress_dense(lr, coef, dict_, 2, 5)) <= bound
    got = host(sr.sr_dict_regress_selected(dev(lr), dev(coef), None, None, dev(dict_), 2, 5, 8))
    assert max_abs_err(got, oracle.dict_regress_selected(lr, coef, None, None, dict_, 2, 5, 8)) <= bound


# ------------------------------------------------------------------ LR pixels that are not finite

# kernel (sr_test_force_kernel; -1 = host rules), mode, n, c, h, w, scale, D, k, coefficients: the kernels that make their
# up-sampled tiles separably, each with more tiles than thread blocks where its tiles follow one another in a block, and those on
# the smallest frames
NON_FINITE_LR = [
    (-1, "dense", 2, 3, 12, 70, 2, 32, 5, "f16"), (-1, "dense", 1, 4, 9, 50, 3, 12, 9, "f32"), (-1, "dense", 1, 1, 20, 131, 1, 40, 3, "f32"),      # the split kernel
    (0, "dense", 2, 3, 12, 70, 2, 32, 5, "f16"),
    (1, "dense", 2, 3, 130, 320, 2, 32, 5, "f16"), (1, "dense", 2, 1, 400, 500, 1, 24, 3, "f16"), (1, "dense", 2, 1, 90, 136, 4, 72, 7, "f16"),
    (1, "fused", 2, 3, 130, 320, 2, 32, 5, "f16"), (1, "compact", 1, 3, 96, 160, 3, 32, 5, "f16"),
    (2, "dense", 2, 3, 130, 320, 2, 16, 5, "f16"), (4, "compact", 2, 3, 130, 320, 2, 32, 5, "f16"),
    (-1, "dense", 2, 3, 130, 321, 2, 16, 5, "f16"), (-1, "dense", 2, 1, 300, 451, 1, 16, 3, "f16"), (-1, "dense", 1, 2, 101, 231, 3, 16, 7, "f16"),
    (-1, "dense", 2, 3, 130, 320, 2, 16, 5, "f32"), (-1, "dense", 2, 1, 300, 451, 1, 8, 3, "f32"), (-1, "dense", 1, 1, 101, 230, 3, 8, 9, "f32"),
    (-1, "fused", 2, 3, 40, 77, 2, 16, 5, "f16"), (-1, "producer", 2, 3, 100, 300, 2, 16, 5, "f16")]


@pytest.mark.parametrize("case", NON_FINITE_LR, ids=lambda c: "-".join(map(str, c)))
def test_a_non_finite_lr_pixel_reaches_only_the_pixels_that_read_it(case):
    kernel, mode, n, c, h, w, r, D, k, dt = case
    wl = sr_inputs.Workload("t", n, c, h, w, r, D=D, k=k, coef_dtype=dt)
    lr, d, coef = sr_inputs.make_inputs(wl)
    d, s, p = signed_asymmetric_dictionary(d, seed=k), 8, (k - 1) // 2
    d[d == 0] = 0.25                                          # every tap reads its pixel
    dco, ddi = dev(coef), dev(d)
    if mode == "dense":
        call = lambda x: sr.sr_dict_regress_dense(x, dco, ddi, r, k)
    elif mode == "fused":
        call = lambda x: sr.sr_dict_regress_selected(x, dco, None, None, ddi, r, k, s)
    elif mode == "compact":
        idx, sel = sr.sr_dict_select(dco, s, want_sel=True)
        call = lambda x: sr.sr_dict_regress_selected(x, sel, idx, None, ddi, r, k, s, sr.SR_COEF_COMPACT)
    else:
        feat, wconv, bias = (dev(a) for a in sr_inputs.make_producer(wl, cin=32, kc=1))
        folded = sr.sr_producer_fold(wconv, bias, ddi, r, k)
        call = lambda x: sr.sr_producer_regress(x, feat, folded, r, k, D, 1)
    sr.sr_test_force_kernel(kernel)
    try:
        clean = host(call(dev(lr)))
        bad, hit = lr.copy(), np.zeros(clean.shape, bool)
        H, W = h * r, w * r
        rng = np.random.default_rng(k)
        spots = [(0, 0, 0), (h - 1, w - 1, 0), (h // 2, 128 // r, 0), (h // 3, 64 // r - 1, n - 1), (h // 3, w - 1, n - 1)]
        spots += [(int(rng.integers(h)), int(rng.integers(w)), int(rng.integers(n))) for _ in range(6)]
        first = lambda Z: (2 * Z + 1 - r) // (2 * r) - 1      # first of the four taps of an HR coordinate
        for j, (y, x, f) in enumerate(spots):
            ch = j % c
            bad[f, ch, y, x] = [np.nan, np.inf, -np.inf][j % 3]
            rows = np.array([any(min(max(first(Z) + a, 0), h - 1) == y for a in range(4)) for Z in range(H)])
            cols = np.array([any(min(max(first(Z) + a, 0), w - 1) == x for a in range(4)) for Z in range(W)])
            near = lambda m, size: np.array([any(m[min(max(Z + a, 0), size - 1)] for a in range(-p, p + 1)) for Z in range(size)])
            hit[f, ch] |= np.outer(near(rows, H), near(cols, W))
        for _ in range(2):                                    # the second call meets blocks that have just worked on such a frame
            out = host(call(dev(bad)))
            np.testing.assert_array_equal(~np.isfinite(out), hit)
            np.testing.assert_array_equal(out[~hit], clean[~hit])
    finally:
        sr.sr_test_force_kernel(-1)


TILE_CASES = [  # k, c, h, w, scale, D: fp32 frames large enough for the register-tiled kernel, every atom size, both copy widths
    (1, 1, 260, 300, 1, 5), (3, 3, 130, 161, 2, 9), (5, 3, 101, 87, 3, 72), (5, 4, 70, 69, 4, 7), (7, 3, 100, 95, 3, 16), (9, 2, 80, 64, 4, 8),
    (5, 3, 97, 100, 3, 20), (5, 2, 280, 281, 1, 2), (7, 3, 100, 125, 3, 16)]


@pytest.mark.parametrize("case", TILE_CASES, ids=lambda c: "-".join(map(str, c)))
def test_register_tiled_fp32_dense_and_subset(case):
    k, c, h, w, r, D = case
    wl = sr_inputs.Workload("tile", 1, c, h, w, r, D=D, k=k, coef_dtype="f32")
    lr, d, coef = sr_inputs.make_inputs(wl)
    # (differences of Gaussians of one tap are 0 / 0: random atoms there)
    d = signed_asymmetric_dictionary(d, seed=k) if k > 1 else np.random.default_rng(k).uniform(-1, 1, d.shape).astype(np.float32)
    assert wl.npix >= 148 * 512
    out = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), r, k))
    assert max_abs_err(out, oracle.dict_regress_dense(lr, coef, d, r, k)) <= TOL_F32
    s = min(D, 3)
    S, gamma = np.arange(D - 1, D - 1 - s, -1).astype(np.uint8), signed_gamma(s)
    want = oracle.dict_regress_selected(lr, coef, S, gamma, d, r, k, s, flags=oracle.IDX_GLOBAL)
    got = host(sr.sr_dict_regress_selected(dev(lr), dev(coef), dev(S), dev(gamma), dev(d), r, k, s, sr.SR_IDX_GLOBAL))
    assert max_abs_err(got, want) <= TOL_F32
    # an unaligned view of the same planes (single-word copies) and the kept planes alone
    room = torch.zeros(coef.size + 4, dtype=torch.float32, device="cuda")
    view = room[1:1 + coef.size].view(coef.shape).copy_(dev(coef))
    np.testing.assert_array_equal(host(sr.sr_dict_regress_dense(dev(lr), view, dev(d), r, k)), out)
    kept = dev(np.ascontiguousarray(coef[:, S]))
    np.testing.assert_array_equal(host(sr.sr_dict_regress_selected(dev(lr), kept, dev(S), dev(gamma), dev(d), r, k, s, sr.SR_IDX_GLOBAL | sr.SR_COEF_COMPACT)), got)


@pytest.mark.parametrize("D", [240, 241, 256])
def test_fp32_9x9_four_channels_with_more_atoms_than_the_register_tiled_kernel_holds(D):
    wl = sr_inputs.Workload("tile", 1, 4, 148, 512, 1, D=D, k=9, coef_dtype="f32")
    lr, d, coef = sr_inputs.make_inputs(wl)
    want = oracle.dict_regress_dense(lr, coef, d, 1, 9)
    assert max_abs_err(host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), 1, 9)), want) <= TOL_F32
    s = D - 1
    S, gamma = np.arange(1, D).astype(np.uint8), signed_gamma(s)
    want = oracle.dict_regress_selected(lr, coef, S, gamma, d, 1, 9, s, flags=oracle.IDX_GLOBAL)
    assert max_abs_err(host(sr.sr_dict_regress_selected(dev(lr), dev(coef), dev(S), dev(gamma), dev(d), 1, 9, s, sr.SR_IDX_GLOBAL)), want) <= TOL_F32


# Batches of patches and frames a few columns wide: their tiles would be mostly empty, so the rules weigh what a tile covers
NARROW = [(80, 32, 32, 1), (19, 32, 32, 2), (3, 300, 31, 3), (1, 2000, 20, 2), (300, 9, 5, 3)]


@pytest.mark.parametrize("dt", ["f16", "f32"])
@pytest.mark.parametrize("n,h,w,r", NARROW)
@pytest.mark.parametrize("k,D", [(3, 5), (5, 24), (7, 17)])
def test_batches_of_narrow_frames(dt, n, h, w, r, k, D):
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("narrow", n, 2, h, w, r, D=D, k=k, coef_dtype=dt))
    d = signed_asymmetric_dictionary(d, seed=k)
    tol = TOL_F32 if dt == "f32" else TOL_F16
    assert max_abs_err(host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), r, k)), oracle.dict_regress_dense(lr, coef, d, r, k)) <= tol
    s = 3
    S, gamma = np.arange(D - 1, D - 1 - s, -1).astype(np.uint8), signed_gamma(s)
    want = oracle.dict_regress_selected(lr, coef, S, gamma, d, r, k, s, flags=oracle.IDX_GLOBAL)
    assert max_abs_err(host(sr.sr_dict_regress_selected(dev(lr), dev(coef), dev(S), dev(gamma), dev(d), r, k, s, sr.SR_IDX_GLOBAL)), want) <= tol


ROW_CASES = [  # k, n, c, h, w, scale, D: binary16 rows of any width; K-steps of 16 atoms and tiles of 64 x 8 on both sides of their edges
    (5, 1, 3, 41, 43, 3, 72), (5, 2, 3, 9, 21, 3, 16), (5, 1, 1, 17, 65, 1, 17), (5, 1, 4, 5, 63, 1, 15), (3, 2, 3, 13, 33, 2, 1), (3, 1, 2, 27, 11, 4, 33),
    (7, 1, 3, 19, 29, 3, 32), (7, 2, 1, 33, 67, 1, 40), (5, 1, 3, 3, 1, 5, 128), (5, 3, 3, 1, 1, 1, 256), (7, 1, 3, 30, 31, 2, 100), (5, 1, 3, 90, 101, 5, 24),
    # both sides of the 32768 pixels from which the row kernel is considered (ROW_KERNEL_CASES are the ones that run it)
    (5, 2, 3, 41, 67, 3, 72), (5, 1, 1, 1, 32767, 1, 15), (5, 1, 1, 1, 32769, 1, 17), (3, 1, 4, 257, 129, 1, 33), (7, 1, 3, 63, 131, 2, 40), (7, 1, 2, 91, 91, 2, 128),
    (3, 2, 3, 65, 67, 2, 1), (5, 1, 2, 33000, 1, 1, 16)]


@pytest.mark.parametrize("case", ROW_CASES, ids=lambda c: "-".join(map(str, c)))
@pytest.mark.parametrize("magnitude", [1.0, 2.0 ** 20, 2.0 ** -30])
@pytest.mark.parametrize("kernel", [-1, 0])                  # the smaller ones: the split kernel, the thread-per-pixel kernel
def test_binary16_rows_of_any_width(case, magnitude, kernel):
    with on_kernel(kernel):
        _binary16_rows_of_any_width(case, magnitude)


def _binary16_rows_of_any_width(case, magnitude):
    k, n, c, h, w, r, D = case
    wl = sr_inputs.Workload("rows", n, c, h, w, r, D=D, k=k)
    lr, d, coef = sr_inputs.make_inputs(wl)
    d = (signed_asymmetric_dictionary(d, seed=k) * np.float32(magnitude)).astype(np.float32)
    # the dictionary enters whole and sums are fp32: within the fp32 bound (D k^2 terms of at most 1.2 in all)
    tol = TOL_F32 * magnitude
    want = oracle.dict_regress_dense(lr, coef, d, r, k)
    out = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), r, k))
    assert max_abs_err(out, want) <= tol
    # tensors that start in the upper half of a word, their last element alone in one
    room = torch.zeros(coef.size + 8, dtype=torch.float16, device="cuda")
    view = room[1:1 + coef.size].view(coef.shape).copy_(dev(coef))
    np.testing.assert_array_equal(host(sr.sr_dict_regress_dense(dev(lr), view, dev(d), r, k)), out)
    s = min(D, 9)                                             # nine: beyond the small-subset kernel
    S, gamma = np.arange(D - 1, D - 1 - s, -1).astype(np.uint8), signed_gamma(s)
    want = oracle.dict_regress_selected(lr, coef, S, gamma, d, r, k, s, flags=oracle.IDX_GLOBAL)
    got = host(sr.sr_dict_regress_selected(dev(lr), view, dev(S), dev(gamma), dev(d), r, k, s, sr.SR_IDX_GLOBAL))
    assert max_abs_err(got, want) <= tol
    kept = dev(np.ascontiguousarray(coef[:, S]))
    np.testing.assert_array_equal(host(sr.sr_dict_regress_selected(dev(lr), kept, dev(S), dev(gamma), dev(d), r, k, s, sr.SR_IDX_GLOBAL | sr.SR_COEF_COMPACT)), got)


@pytest.mark.parametrize("k,n,h,w,D", [(5, 2, 301, 257, 48), (7, 2, 211, 97, 16), (3, 2, 400, 257, 128)])
def test_binary16_rows_that_start_at_any_half_of_a_chunk(k, n, h, w, D):
    # the tensor's first chunk begins up to fourteen bytes in front of it; those bytes are not the tensor's
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("rows", n, 1, h, w, 1, D=D, k=k))
    S = np.arange(D, dtype=np.uint8)
    room = torch.zeros(coef.size + 16, dtype=torch.float16, device="cuda")
    first = None
    for start in range(8):
        room.fill_(float("nan"))
        view = room[start:start + coef.size].view(coef.shape).copy_(dev(coef))
        got = host(sr.sr_dict_regress_dense(dev(lr), view, dev(d), 1, k))
        first = got if first is None else first
        np.testing.assert_array_equal(got, first)
        np.testing.assert_array_equal(host(sr.sr_dict_regress_selected(dev(lr), view, dev(S), None, dev(d), 1, k, D, sr.SR_IDX_GLOBAL)), first)
    assert max_abs_err(first, oracle.dict_regress_dense(lr, coef, d, 1, k)) <= TOL_F32


# k, n, c, h, w, scale, D: frames that the rules give to the row kernel (by its estimated time; none of those above is large or
# has atoms enough). K-steps and 64-pixel columns on both sides of their edges, one to four channels, one to three rows a
# warp; the last four with more tiles than blocks, so that a block works on several (k = 3, 5, 7, two and five K-steps)
ROW_KERNEL_CASES = [
    (5, 2, 4, 211, 129, 1, 16), (5, 1, 2, 161, 43, 3, 31), (5, 2, 3, 97, 43, 3, 33), (5, 1, 3, 97, 65, 3, 48), (5, 2, 1, 129, 85, 2, 49),
    (5, 2, 2, 97, 65, 2, 256), (3, 2, 3, 97, 85, 2, 48), (3, 2, 3, 129, 43, 3, 65), (3, 2, 4, 97, 85, 2, 200), (7, 2, 3, 97, 65, 3, 3),
    (7, 2, 1, 211, 97, 1, 16), (7, 2, 4, 85, 85, 2, 17), (7, 2, 3, 161, 161, 1, 33), (7, 1, 2, 201, 97, 2, 100),
    (3, 1, 3, 160, 401, 3, 72), (7, 1, 2, 151, 151, 3, 40), (5, 1, 3, 213, 321, 3, 72), (5, 2, 3, 201, 321, 1, 24)]


@pytest.mark.parametrize("case", ROW_KERNEL_CASES, ids=lambda c: "-".join(map(str, c)))
def test_row_kernel_dense_and_gathered(case):
    k, n, c, h, w, r, D = case
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("rows", n, c, h, w, r, D=D, k=k))
    d = signed_asymmetric_dictionary(d, seed=k)
    out = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), r, k))
    assert max_abs_err(out, oracle.dict_regress_dense(lr, coef, d, r, k)) <= TOL_F32
    # more than three K-steps where there are as many atoms
    s = min(D, 61) - (D > 20)
    S, gamma = np.arange(D - 1, D - 1 - s, -1).astype(np.uint8), signed_gamma(s)
    want = oracle.dict_regress_selected(lr, coef, S, gamma, d, r, k, s, flags=oracle.IDX_GLOBAL)
    # (signed weights up to 1.5 on up to 60 atoms of up to 1 / D each)
    assert max_abs_err(host(sr.sr_dict_regress_selected(dev(lr), dev(coef), dev(S), dev(gamma), dev(d), r, k, s, sr.SR_IDX_GLOBAL)), want) <= 2 * TOL_F32
    kept = dev(np.ascontiguousarray(coef[:, S]))
    assert max_abs_err(host(sr.sr_dict_regress_selected(dev(lr), kept, dev(S), dev(gamma), dev(d), r, k, s, sr.SR_IDX_GLOBAL | sr.SR_COEF_COMPACT)), want) <= 2 * TOL_F32


@pytest.mark.parametrize("k,D", [(3, 72), (5, 53), (7, 33)])
@pytest.mark.parametrize("flags", [0, sr.SR_CLAMP01 | sr.SR_OUT_U8])
def test_row_kernel_with_coefficients_that_are_not_finite(k, D, flags):
    # beside the edges of a 64-pixel column and of a row, in the first, the last and an inner atom: the same infinities and NaN
    # as the sum has, in that pixel alone
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("rows", 2, 3, 97, 85, 2, D=D, k=k))
    d = signed_asymmetric_dictionary(d, seed=k)
    d[D - 1] = np.abs(d[D - 1]) + 0.01                        # with finite taps of one sign: an infinity, not NaN
    args = (dev(d), 2, k, flags)
    clean = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), *args))
    bad, hit = coef.copy(), np.zeros(clean.shape, bool)
    for j, (f, y, x) in enumerate([(0, 0, 0), (0, 30, 63), (0, 30, 64), (0, 31, 65), (1, 100, 169), (1, 101, 0), (1, 193, 169), (0, 7, 127), (1, 8, 128), (0, 60, 150), (0, 61, 150)]):
        bad[f, [D - 1, 0, D // 2][j % 3], y, x] = [np.inf, -np.inf, np.nan, np.inf][j % 4]
        hit[f, :, y, x] = True
    out = host(sr.sr_dict_regress_dense(dev(lr), dev(bad), *args))
    np.testing.assert_array_equal(out[~hit], clean[~hit])
    want = oracle.dict_regress_dense(lr, bad, d, 2, k, flags=flags & 1)[hit]
    if flags == 0:
        np.testing.assert_array_equal(np.isnan(out[hit]), np.isnan(want))
        np.testing.assert_array_equal(out[hit][~np.isnan(want)], want[~np.isnan(want)].astype(np.float32))
        assert np.isinf(want).any() and np.isnan(want).any()
    else:                                                     # NaN is stored as 0, as by the other kernels
        np.testing.assert_array_equal(out[hit], np.where(np.isnan(want), 0, np.clip(want, 0, 1) * 255))


@pytest.mark.parametrize("magnitude", [2.0 ** 120, 2.0 ** -122])
def test_row_kernel_at_the_ends_of_the_dictionary_range(magnitude):
    lr, d, coef = sr_inputs.make_inputs(sr_inputs.Workload("rows", 1, 3, 97, 65, 3, D=48, k=5))
    d = (signed_asymmetric_dictionary(d, seed=5) * np.float32(magnitude)).astype(np.float32)
    got = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), 3, 5)).astype(np.float64) / magnitude
    want = oracle.dict_regress_dense(lr, coef, d, 3, 5) / magnitude
    # (2^-122: results below 2^-126 keep 2^-149, here 2^-27)
    assert np.abs(got - want).max() <= TOL_F32


@pytest.mark.parametrize("kernel", [-1, 0])                  # a small frame: the split kernel, the thread-per-pixel kernel
def test_binary16_rows_keep_a_non_finite_coefficient_to_its_pixel(kernel):
    with on_kernel(kernel):
        _keep_a_non_finite_coefficient()


def _keep_a_non_finite_coefficient():
    wl = sr_inputs.Workload("rows", 1, 3, 20, 27, 3, D=20, k=5)
    lr, d, coef = sr_inputs.make_inputs(wl)
    clean = host(sr.sr_dict_regress_dense(dev(lr), dev(coef), dev(d), 3, 5))
    bad = coef.copy()
    bad[0, 7, 30, 40] = np.inf
    bad[0, 19, 31, 80] = np.nan
    out = host(sr.sr_dict_regress_dense(dev(lr), dev(bad), dev(d), 3, 5))
    hit = np.zeros(out.shape, bool)
    hit[:, :, 30, 40] = hit[:, :, 31, 80] = True
    np.testing.assert_array_equal(out[~hit], clean[~hit])
    assert not np.isfinite(out[hit]).any()
