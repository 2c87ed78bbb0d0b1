"""The dictionary selection search (Section III-A, Algorithm 1) on the GPU against the oracle: the Gram statistics
within the fp32 bound of their 32-pixel partial sums, the search bit for bit on identical statistics (same kept atoms,
same lambda path, same losses), and the two together end to end into the global-subset regression."""
import numpy as np
import pytest
import torch

import oracle
import paper_2303_08999_b200 as sr
import sr_inputs
from gpu_util import TOL_F16, dev, host, signed_asymmetric_dictionary
from test_oracle_pins_selection import DEAD

pytestmark = pytest.mark.gpu


def _problem(D, k, r, h, w, dt="f16", n=1, c=3, seed=0, planted=None):
    wl = sr_inputs.Workload("t", n, c, h, w, r, D=D, k=k, coef_dtype=dt)
    lr, d, coef = sr_inputs.make_inputs(wl, seed=sr_inputs.BASE_SEED + seed)
    d = signed_asymmetric_dictionary(d, seed=seed) if k > 1 else np.random.default_rng(seed).uniform(-1, 1, d.shape).astype(np.float32)
    if planted is not None:                                   # a few atoms carry most of the coefficient energy
        scale = np.full(D, 0.03, np.float32)
        scale[planted] = 1.0
        coef = (coef.astype(np.float32) * scale[None, :, None, None]).astype(coef.dtype)
    rng = np.random.default_rng(seed + 1)
    target = (oracle.dict_regress_dense(lr, coef, d, r, k) + rng.normal(0, 0.01, (n, c, h * r, w * r))).astype(np.float32)
    return wl, lr, d, coef, target


def _gram_close(got, want_G, want_b, want_hh):
    G, b, hh = (host(t) for t in got)
    dg = np.sqrt(np.diag(want_G))
    assert np.all(np.abs(G - want_G) <= 2e-5 * np.outer(dg, dg) + 1e-30)
    assert np.all(np.abs(b - want_b) <= 2e-5 * dg * np.sqrt(want_hh) + 1e-30)
    assert abs(hh[0] - want_hh) <= 1e-6 * want_hh
    np.testing.assert_array_equal(G, G.T)                    # both triangles are summed from the same products


@pytest.mark.parametrize("D,k,r,h,w,dt,n,c", [(72, 5, 4, 10, 12, "f16", 1, 3), (16, 3, 2, 9, 7, "f32", 2, 3), (128, 7, 3, 6, 8, "f16", 1, 1),
                                              (7, 1, 2, 5, 5, "f16", 1, 2), (33, 5, 2, 8, 8, "f16", 1, 3)])
def test_gram_statistics_match_the_oracle(D, k, r, h, w, dt, n, c):
    wl, lr, d, coef, target = _problem(D, k, r, h, w, dt, n, c)
    want = oracle.selection_gram(lr, coef, d, target, None, r, k)
    _gram_close(sr.sr_selection_gram(dev(lr), dev(coef), dev(d), dev(target), None, r, k), *want)
    # a sample with repeats and out-of-range entries (those are skipped), not a multiple of the 32-pixel chunk
    rng = np.random.default_rng(2)
    samples = rng.integers(0, wl.npix, size=77, dtype=np.int64)
    samples[5] = samples[6]
    want = oracle.selection_gram(lr, coef, d, target, samples, r, k)
    with_bad = np.concatenate([samples, np.array([-1, wl.npix, 1 << 40], dtype=np.int64)])
    _gram_close(sr.sr_selection_gram(dev(lr), dev(coef), dev(d), dev(target), dev(with_bad), r, k), *want)
    # the bilinear form of stage 1, and twice the same call gives the same bits
    want = oracle.selection_gram(lr, coef, d, target, None, r, k, flags=oracle.UPSAMPLE_BILINEAR)
    a = sr.sr_selection_gram(dev(lr), dev(coef), dev(d), dev(target), None, r, k, sr.SR_UPSAMPLE_BILINEAR)
    _gram_close(a, *want)
    b = sr.sr_selection_gram(dev(lr), dev(coef), dev(d), dev(target), None, r, k, sr.SR_UPSAMPLE_BILINEAR)
    assert all(torch.equal(x, y) for x, y in zip(a, b))


SEARCHES = [  # D, alpha, delta_alpha, eps
    (24, 0.25, 0.125, 0.05), (16, 0.5, 0.25, 0.0), (72, 0.125, 0.125, 0.02), (40, 0.1, 0.3, 0.0), (9, 1.0 / 3, 1.0 / 3, 0.0)]


@pytest.mark.parametrize("D,alpha,dalpha,eps", SEARCHES)
def test_search_is_bit_identical_on_identical_statistics(D, alpha, dalpha, eps):
    wl, lr, d, coef, target = _problem(D, 3, 2, 10, 10, seed=D)
    G, b, hh = oracle.selection_gram(lr, coef, d, target, None, 2, 3)
    nrows = wl.npix * wl.c
    kw = dict(tol=1e-9, max_sweeps=2000, max_bisect=30)
    want_idx, want_gamma, want_trace = oracle.selection_search(G, b, hh, nrows, alpha, dalpha, eps, 1e-9, **kw)
    idx, gamma, trace = sr.sr_selection_search(dev(G), dev(b), dev(np.array([hh])), nrows, alpha, dalpha, eps, 1e-9, **kw)
    np.testing.assert_array_equal(host(idx), want_idx)
    np.testing.assert_array_equal(host(trace), want_trace)    # alpha_t, lambda, atoms kept, both losses, solves: same bits
    np.testing.assert_array_equal(host(gamma), want_gamma.astype(np.float32))


def test_search_on_orthogonal_features_and_a_singular_refit():
    rng = np.random.default_rng(4)
    n, L = 256, 16
    Q, _ = np.linalg.qr(rng.normal(size=(n, L)))
    Z = Q * rng.uniform(0.5, 2.0, L)
    h = Z @ (rng.permutation(np.linspace(0.2, 3.0, L)) * rng.choice([-1, 1], L)) + 0.01 * rng.normal(size=n)
    G, b, hh = Z.T @ Z, Z.T @ h, h @ h
    want = oracle.selection_search(G, b, hh, n, 0.25, 0.125, 0.0, 1e-6, tol=1e-9, max_sweeps=2000)
    idx, gamma, trace = sr.sr_selection_search(dev(G), dev(b), dev(np.array([hh])), n, 0.25, 0.125, 0.0, 1e-6)
    np.testing.assert_array_equal(host(idx), want[0])
    np.testing.assert_array_equal(host(trace), want[2])
    # an atom that never responds (zero row and column of G) cannot be dropped by the LASSO and makes the re-fit
    # singular: both sides report it instead of returning numbers
    G0, b0 = np.diag([1.0, 2.0, 0.0, 3.0]), np.array([1.0, 1.5, 0.0, 2.0])
    with pytest.raises(ValueError):
        oracle.selection_search(G0, b0, 5.0, 10, 0.75, 0.25, 0.0, 1e-3)
    with pytest.raises(sr.SrError):
        sr.sr_selection_search(dev(G0), dev(b0), dev(np.array([5.0])), 10, 0.75, 0.25, 0.0, 1e-3)


def test_search_end_to_end_finds_planted_atoms_and_feeds_the_subset_regression():
    planted = np.array([3, 17, 29, 41, 50, 58, 63, 70])
    wl, lr, d, coef, target = _problem(72, 5, 4, 24, 32, planted=planted)
    dlr, dco, ddi, dta = dev(lr), dev(coef), dev(d), dev(target)
    rng = np.random.default_rng(8)
    samples = np.sort(rng.choice(wl.npix, size=4000, replace=False)).astype(np.int64)    # the paper samples its LASSO features
    G, b, hh = sr.sr_selection_gram(dlr, dco, ddi, dta, dev(samples), 4, 5)
    nrows = samples.size * wl.c
    idx, gamma, trace = sr.sr_selection_search(G, b, hh, nrows, 8 / 72, 16 / 72, 0.0, 1e-9)
    oG, ob, ohh = oracle.selection_gram(lr, coef, d, target, samples, 4, 5)
    want_idx, want_gamma, want_trace = oracle.selection_search(oG, ob, ohh, nrows, 8 / 72, 16 / 72, 0.0, 1e-9, tol=1e-9, max_sweeps=2000)
    np.testing.assert_array_equal(host(idx), planted)
    np.testing.assert_array_equal(want_idx, planted)
    assert np.abs(host(gamma) - want_gamma).max() <= 1e-3 * np.abs(want_gamma).max()
    np.testing.assert_array_equal(host(trace)[:, 2], want_trace[:, 2])
    # the search's output is the input of the paper's inference-time rule
    out = sr.sr_dict_regress_selected(dlr, dco, idx.contiguous(), gamma.contiguous(), ddi, 4, 5, 8, sr.SR_IDX_GLOBAL)
    want = oracle.dict_regress_selected(lr, coef, host(idx), host(gamma), d, 4, 5, 8, flags=oracle.IDX_GLOBAL)
    assert np.abs(host(out) - want).max() <= TOL_F16
    assert np.mean((host(out) - target) ** 2) <= 0.03 * np.mean(target.astype(np.float64) ** 2)   # eight atoms of 72 keep the image
    assert sr.sr_device_status() == 0


@pytest.mark.parametrize("D,k,r,h,w,dt,n,c,base", [(32, 3, 2, 9, 7, "f16", 1, 3, 0), (33, 5, 3, 7, 9, "f16", 2, 3, 0), (72, 5, 3, 7, 5, "f16", 1, 1, 2),
                                                   (71, 7, 1, 9, 13, "f16", 1, 4, 0), (128, 9, 8, 2, 3, "f32", 1, 2, 0), (8, 3, 2, 5, 5, "f32", 3, 16, 0)])
def test_gram_at_block_edges_and_odd_planes(D, k, r, h, w, dt, n, c, base):
    # both block sizes on both sides of their atom limits, odd plane sizes (a binary16 coefficient in either half of its
    # word, with the tensor's first or last element alone in one), more channels than a chunk has groups of rows
    wl, lr, d, coef, target = _problem(D, k, r, h, w, dt, n, c, seed=D)
    co = dev(coef)
    if base:                                                  # a tensor that starts in the upper half of a word
        room = torch.zeros(co.numel() + 8, dtype=co.dtype, device="cuda")
        co = room[1:1 + co.numel()].view(co.shape).copy_(co)
        assert co.data_ptr() % 4 == 2
    _gram_close(sr.sr_selection_gram(dev(lr), co, dev(d), dev(target), None, r, k), *oracle.selection_gram(lr, coef, d, target, None, r, k))


@pytest.mark.parametrize("D", [16, 33, 72, 128])
@pytest.mark.parametrize("n,h,w", [(1, 120, 100), (1, 9, 11)])
def test_gram_adds_at_most_the_terms_of_32_pixels_in_fp32(D, n, h, w):
    # responses that are all the same number, whose multiples have no room in fp32: m terms added one after the other are off by at
    # most (m + 1) / 2 units of 2^-24, and with this number 80 terms are off by 20
    v = np.float16(1.251953125)
    lr, coef, d = np.ones((n, 1, h, w), np.float32), np.full((n, D, h, w), v, np.float16), np.ones((D, 1), np.float32)
    target = np.full((n, 1, h, w), np.float32(v))
    G, b, hh = (host(x) for x in sr.sr_selection_gram(dev(lr), dev(coef), dev(d), dev(target), None, 1, 1))
    want = n * h * w * float(v) ** 2
    for got in (G, b, hh):
        assert np.abs(got - want).max() <= 16.5 * 2.0 ** -24 * want


@pytest.mark.parametrize("D", [1, 7, 8, 9, 31, 33, 64, 65, 97, 128])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -700, 2.0 ** 640])
def test_search_bits_at_block_edges_and_extreme_scales(D, scale):
    # coordinate blocks of eight, residuals in registers of 32: both sides of their edges; statistics scaled by a power of
    # two lie outside the range of the fast quotient, so the same path has to be walked with the library's division
    rng = np.random.default_rng(D)
    n = 4 * D + 20
    Z = rng.normal(size=(n, D)) * np.exp(-3.0 * rng.permutation(D) / D)
    h = Z.sum(1) + 0.05 * rng.normal(size=n)
    G, b, hh = (Z.T @ Z) * scale, (Z.T @ h) * scale, (h @ h) * scale
    G = (G + G.T) / 2
    alpha, dalpha = max(1, D // 4) / D, max(1, D // 3) / D
    kw = dict(tol=1e-9, max_sweeps=300, max_bisect=20)
    want_idx, want_gamma, want_trace = oracle.selection_search(G, b, hh, n, alpha, dalpha, 0.0, 1e-6 * scale, **kw)
    idx, gamma, trace = sr.sr_selection_search(dev(G), dev(b), dev(np.array([hh])), n, alpha, dalpha, 0.0, 1e-6 * scale, **kw)
    np.testing.assert_array_equal(host(idx), want_idx)
    np.testing.assert_array_equal(host(trace), want_trace)
    np.testing.assert_array_equal(host(gamma), want_gamma.astype(np.float32))


@pytest.mark.parametrize("diag", DEAD, ids=len)
@pytest.mark.parametrize("lambda0", [1e-3, 5e-324, np.inf])
def test_search_ends_when_no_lambda_removes_enough_atoms(diag, lambda0):
    b = np.where(np.array(diag) > 0, 1.0, 0.0)
    with pytest.raises(sr.SrError):
        sr.sr_selection_search(dev(np.diag(diag)), dev(b), dev(np.array([5.0])), 10, 0.25, 0.25, 0.0, lambda0)


@pytest.mark.parametrize("D", [7, 8, 31, 33, 64, 65, 96, 97, 128])
@pytest.mark.parametrize("max_bisect", [1, 4, 5, 6, 30])
def test_search_bits_over_atoms_and_bisections(D, max_bisect):
    # sizes on both sides of the warp's rows of 32 coordinates and the blocks of eight; bisections on both sides of a tree of five levels
    rng = np.random.default_rng(D)
    Z = rng.normal(size=(600, D)) * np.exp(-3.0 * rng.permutation(D) / D) + 0.1 * rng.normal(size=(600, 1))
    h = Z.sum(1) + 0.05 * rng.normal(size=600)
    G, b, hh = Z.T @ Z, Z.T @ h, h @ h
    args = (600.0, 0.25, 0.3, 0.0, 1e-7)
    want = oracle.selection_search(G, b, hh, *args, tol=1e-9, max_sweeps=500, max_bisect=max_bisect)
    idx, gamma, trace = sr.sr_selection_search(dev(G), dev(b), dev(np.array([hh])), *args, tol=1e-9, max_sweeps=500, max_bisect=max_bisect)
    np.testing.assert_array_equal(host(idx), want[0])
    np.testing.assert_array_equal(host(trace), want[2])
    np.testing.assert_array_equal(host(gamma), want[1].astype(np.float32))


def test_search_where_a_quotient_lies_next_to_the_middle_of_two_numbers():
    # 1 / (1 - 2^-53) = 1 + 2^-53 + 2^-106: the quotient made from the rounded reciprocal and its remainder is off by one unit, and the
    # sweep is made again by division; hh makes the loss the difference of the two
    G, b = np.diag([1.0 - 2.0 ** -53, 4.0]), np.array([2.0, 0.5])
    hh = 2 * b[0] * 1.0 - G[0, 0]
    want = oracle.selection_search(G, b, hh, 2, 0.5, 0.5, 0.0, 1.0, tol=1e-9, max_sweeps=50)
    idx, gamma, trace = sr.sr_selection_search(dev(G), dev(b), dev(np.array([hh])), 2, 0.5, 0.5, 0.0, 1.0, max_sweeps=50)
    np.testing.assert_array_equal(host(idx), want[0])
    np.testing.assert_array_equal(host(trace), want[2])


@pytest.mark.parametrize("e", [1, 10, 20, 30, 40, 46, 50])
def test_search_bits_where_residuals_lie_just_above_the_threshold(e):
    # numerators of about 2^-e of the threshold: what the quick quotient rounds away grows with 2^e against the quotient
    rng = np.random.default_rng(e)
    D = 12
    off = np.triu(rng.uniform(-0.02, 0.02, (D, D)), 1)
    G = np.diag(rng.uniform(1, 2, D)) + off + off.T
    b = np.full(D, 0.5)
    b[::2] = 1 + rng.uniform(1, 2, D // 2) * 2.0 ** -e
    args = (2.0, 0.5, 0.5, 0.0, 1.0)
    want = oracle.selection_search(G, b, 0.0, *args, tol=1e-30, max_sweeps=200)
    idx, gamma, trace = sr.sr_selection_search(dev(G), dev(b), dev(np.array([0.0])), *args, tol=1e-30, max_sweeps=200)
    assert len(want[0]) == D // 2
    np.testing.assert_array_equal(host(idx), want[0])
    np.testing.assert_array_equal(host(trace), want[2])
    np.testing.assert_array_equal(host(gamma), want[1].astype(np.float32))
