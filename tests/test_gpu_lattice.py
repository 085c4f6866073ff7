"""GPU parity where the histogram behind the error curve can go wrong: bins taken in windows (many candidates, a grid that
ends far below max|x|), grids that reach beyond max|x|, steps near the smallest normal number, one candidate, one value,
and the row lengths at which the mapping of rows to threads changes.  Same acceptance rule as the other parity tests."""
import numpy as np
import pytest

from paper_1902_06822_b200 import synth
from parity import check_rows

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,k,bits,signed,n_cand,hi_frac,scale", [
    (5, 700, 4, True, 4096, 1.0 / 7, 1.0),          # 57,344 bins, both signs, in windows
    (5, 700, 4, False, 4096, 1.0 / 15, 1.0),
    (3, 9001, 8, True, 4096, 1.0 / 127, 1.0),
    (4, 300, 2, True, 4096, 1e-3, 1.0),             # most values beyond the last threshold of every candidate
    (3, 300, 8, True, 4096, 1e-36, 1.0),            # ... by more than binary32 holds
    (3, 300, 4, True, 4096, 1e-37, 2.0 ** 50),
    (2000, 300, 8, True, 4096, 1e-36, 1.0),
    (4, 28672, 3, True, 4096, 1.0, 1.0),            # the longest row with the most candidates
    (6, 500, 4, True, 256, 3.0, 1.0),               # fewer bins than candidates
    (6, 500, 4, True, 1000, 40.0, 1.0),
    (6, 500, 4, True, 512, 1.0, 2.0 ** -112),       # step below 1e-30, reciprocals would overflow without scaling
    (6, 500, 3, True, 64, 1.0, 2.0 ** 59),          # the sum of squares overflows binary32
    (7, 1, 4, True, 1, 1.0, 1.0),
    (9, 33, 8, True, 7, 1.0, 1.0),
    (2500, 33, 4, True, 1000, 1.0, 1.0),            # lanes per row: two; long rows of the same path
    (2500, 896, 4, True, 1024, 1.0, 1.0),
    (2500, 897, 4, True, 1024, 1.0, 1.0),
    (2500, 193, 4, True, 1024, 1.0, 2.0 ** -112),   # values scaled, squares would underflow ...
    (2500, 191, 2, True, 300, 0.5, 2.0 ** 59),      # ... or overflow
    (2500, 100, 3, True, 4096, 2.0, 1.0),           # coarse candidates beyond max|x|, wide neighbourhood of the minimum
    (2500, 70, 2, True, 4096, 1.0, 1.0),            # ... of more candidates than are kept
    (151_600, 9, 4, True, 1024, 1.0, 1.0),          # one lane per row: even and odd lengths,
    (151_600, 17, 4, False, 300, 1.0, 1.0),         # a last unit that is not full
    (151_553, 32, 8, True, 64, 1.0, 1.0),
    (2500, 147, 3, True, 1300, 1.0 / 3, 1.0),
])
def test_bins_of_every_kind(s, k, bits, signed, n_cand, hi_frac, scale):
    import gpu_util
    w = synth.student_t3(s * k, seed=77, tensor_id=k).reshape(s, k) * np.float32(scale)
    if not signed:
        w = np.abs(w)
    alpha, sse, idx, q, pk = gpu_util.quantize_weights(w, bits, signed, n_cand, hi_frac, 3, True, bits <= 4)
    rows = np.unique(np.concatenate([np.arange(0, s, max(1, s // 40)), [s - 1]]))
    st = check_rows(w, alpha, sse, idx, q, pk, bits, signed, n_cand, hi_frac, 3, rows=rows)
    assert st["idx_diff"] <= max(1, st["rows"] // 100) and st["alpha_bitwise"] >= 0.99, st


@pytest.mark.parametrize("s,k,bits,packed", [
    (9601, 1, 4, True), (9601, 4, 2, False), (9601, 5, 3, True), (9601, 31, 4, True),       # one lane per row ...
    (9601, 32, 4, True), (9601, 33, 4, True), (9601, 64, 3, False), (9601, 65, 4, False),   # ... two, four,
    (9601, 127, 4, True), (9601, 129, 8, False), (3001, 256, 4, True), (3001, 257, 4, True),
    (1601, 512, 2, True), (1601, 513, 4, True), (1301, 1023, 4, True), (1301, 1024, 4, False),   # ... all of a warp
    (1301, 1025, 4, True),                                                                  # one value more: block per row
    (700, 3, 4, True), (701, 160, 4, True), (700, 161, 8, False),                           # few rows: candidate per lane, block
])
def test_short_rows_by_lanes(s, k, bits, packed):
    import gpu_util
    w = synth.student_t3(s * k, seed=85, tensor_id=k).reshape(s, k)
    alpha, sse, idx, q, pk = gpu_util.quantize_weights(w, bits, True, 700, 1.0, 3, True, packed)
    rows = np.unique(np.concatenate([np.arange(0, s, max(1, s // 60)), np.arange(s - 40, s)]))
    st = check_rows(w, alpha, sse, idx, q, pk, bits, True, 700, 1.0, 3, rows=rows)
    assert st["idx_diff"] <= max(1, st["rows"] // 100) and st["alpha_bitwise"] >= 0.98, st


@pytest.mark.parametrize("s,k,bits,n_cand", [
    (9601, 27, 3, 1024), (9601, 27, 8, 720), (3001, 300, 8, 1008), (701, 40, 4, 720), (1601, 576, 2, 1024),
])
def test_rows_whose_largest_value_divides_evenly(s, k, bits, n_cand):
    """Equal errors at every candidate that divides the one large value: few enough to be listed, and too many."""
    import gpu_util
    w = 1e-4 * synth.student_t3(s * k, seed=89, tensor_id=k).reshape(s, k)
    w[:, k // 2] = np.where(np.arange(s) % 2, np.float32(3.0), np.float32(-1e4))
    alpha, sse, idx, q, pk = gpu_util.quantize_weights(w, bits, True, n_cand, 1.0, 3, True, False)
    rows = np.unique(np.concatenate([np.arange(0, s, max(1, s // 40)), [s - 1]]))
    st = check_rows(w, alpha, sse, idx, q, None, bits, True, n_cand, 1.0, 3, rows=rows)
    assert st["idx_diff"] <= max(1, st["rows"] // 100) and st["alpha_bitwise"] >= 0.98, st


@pytest.mark.parametrize("k", [897, 1027, 4098, 25087])
@pytest.mark.parametrize("packed", [False, True])
def test_rows_of_ragged_length(k, packed):
    """Rows that start at every offset from 16 bytes and whose codes do not fill whole words."""
    import gpu_util
    w = synth.student_t3(7 * k, seed=81, tensor_id=k).reshape(7, k)
    alpha, sse, idx, q, pk = gpu_util.quantize_weights(w, 4, True, 300, 1.0, 3, True, packed)
    st = check_rows(w, alpha, sse, idx, q, pk, 4, True, 300, 1.0, 3)
    assert st["idx_diff"] == 0 and st["alpha_bitwise"] >= 0.85, st      # a scale at a rounding boundary may differ in one row of 7


@pytest.mark.parametrize("k,bits,n_cand,constant", [
    (25087, 4, 1024, False), (25088, 8, 1000, False), (24580, 2, 1024, False), (24580, 4, 1024, True),
])
def test_counts_of_16_bits(k, bits, n_cand, constant):
    """More rows than SMs, of a length that leaves room for two blocks per SM only with 16-bit counts; all values in one bin."""
    import gpu_util
    w = synth.student_t3(330 * k, seed=87, tensor_id=k).reshape(330, k)
    if constant:
        w = np.where(w < 0, np.float32(-0.75), np.float32(0.75))
        w[:, 0] = 1.0
    alpha, sse, idx, q, pk = gpu_util.quantize_weights(w, bits, True, n_cand, 1.0, 3, True, False)
    st = check_rows(w, alpha, sse, idx, q, pk, bits, True, n_cand, 1.0, 3, rows=np.array([0, 163, 329]))
    assert st["idx_diff"] == 0 and st["alpha_bitwise"] >= 0.66, st      # a scale at a rounding boundary may differ in one row of 3


def test_extra_negative_level_decides():
    """Rows whose large values are all negative (or all positive): the two sides of a signed range differ by one code."""
    import gpu_util
    w = synth.student_t3(40 * 600, seed=78).reshape(40, 600)
    w[:20] = -np.abs(w[:20])
    w[20:] = np.abs(w[20:])
    for bits in (2, 3, 4, 8):
        alpha, sse, idx, q, pk = gpu_util.quantize_weights(w, bits, True, 1024, 1.0, 3, True, False)
        st = check_rows(w, alpha, sse, idx, q, None, bits, True, 1024, 1.0, 3)
        assert st["idx_diff"] <= 1 and st["alpha_bitwise"] >= 0.97, (bits, st)


@pytest.mark.parametrize("n,bits,signed,n_cand,hi_frac,scale", [
    (5, 4, True, 7, 1.0, 1.0),                      # one kernel for the whole search: less than a block ...
    (2049, 2, True, 1024, 1.0, 1.0),                # ... two blocks, the second with one value; most candidates
    (303_106, 8, True, 1000, 1.0, 1.0),             # ... every SM, two values over a multiple of four
    (70_001, 4, False, 64, 1.0, 2.0 ** -112),       # step below 1e-30
    (70_001, 4, True, 1025, 1.0, 1.0),              # pipeline of kernels: one candidate more
    (70_001, 4, True, 4096, 1.0 / 7, 1.0),          # bins in windows, none above the last threshold
    (30_000, 8, False, 4096, 1.0 / 100, 1.0),       # ... many windows
    (30_000, 4, True, 1500, 1e-2, 1.0),             # values beyond the last threshold on both sides
    (66_000, 3, True, 64, 5.0, 1.0),                # fewer bins than candidates
    (20_001, 4, True, 4096, 0.9999, 1.0),           # one bin more than a block keeps
    (9_001, 8, False, 4096, 1.0 / 300, 1.0),        # more bins than the workspace holds at once
    (9_001, 8, True, 4096, 1.0 / 300, 1.0),
])
def test_per_tensor_searches_of_every_kind(n, bits, signed, n_cand, hi_frac, scale):
    import gpu_util
    from oracle import omse_oracle as orc
    x = synth.student_t3(n, seed=79, tensor_id=n % 89) * np.float32(scale)
    if not signed:
        x = np.abs(x)
    alpha, sse, idx, curve = gpu_util.activation_scale(x, bits, signed, n_cand, hi_frac, 3)
    ref = orc.activation_scale(x, bits, signed, n_cand, hi_frac, 3)
    ok = ref.sse_curve > 1e-300
    np.testing.assert_allclose(curve[ok], ref.sse_curve[ok], rtol=2e-6)
    if idx != ref.best_idx:
        assert abs(ref.sse_curve[idx] - ref.sse_curve[ref.best_idx]) <= 1e-6 * ref.sse_curve[ref.best_idx]
        ref = orc.phi(x, bits, signed, n_cand, hi_frac, 3, start_idx=idx, want_codes=False)
    assert alpha == pytest.approx(ref.alpha, rel=1e-5, abs=0)
    # the error is a binary32 output: below its normal numbers (1.2e-38) it loses digits and then reads as 0
    assert sse == pytest.approx(ref.sse, rel=1e-5, abs=1e-37)


@pytest.mark.parametrize("n,bits,signed,n_cand,hi_frac", [
    (50_003, 8, False, 2048, 0.3), (50_003, 8, True, 2048, 0.01), (9_001, 4, True, 1000, 0.02), (9_001, 8, False, 2048, 0.004),
])
@pytest.mark.parametrize("values", ["uniform", "mostly_at_the_end"])
def test_grids_below_the_largest_value(n, bits, signed, n_cand, hi_frac, values):
    """Most values lie above the bins that a block keeps, spread out or equal; both workspaces."""
    import torch

    import gpu_util
    from oracle import omse_oracle as orc
    from paper_1902_06822_b200 import binding
    rng = np.random.default_rng(n + bits)
    x = rng.random(n, np.float32) if values == "uniform" else np.where(rng.random(n) < 0.7, 1.0, rng.random(n)).astype(np.float32)
    x = np.where(rng.random(n) < 0.4, -x, x).astype(np.float32) if signed else x
    ref = orc.activation_scale(x, bits, signed, n_cand, hi_frac, 3)
    out = gpu_util.activation_scale(x, bits, signed, n_cand, hi_frac, 3)
    d_x, d = torch.from_numpy(x).cuda(), torch.zeros(2, device="cuda")
    d_idx, d_curve = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(n_cand, dtype=torch.float64, device="cuda")
    binding.omse_activation_scale_static(d_x, n, bits, signed, n_cand, hi_frac, 3, d[:1], d[1:], d_idx, d_curve)
    for alpha, sse, idx, curve in (out, (d[0].item(), d[1].item(), d_idx.item(), d_curve.cpu().numpy())):
        np.testing.assert_allclose(curve, ref.sse_curve, rtol=2e-6)
        assert idx == ref.best_idx or abs(ref.sse_curve[idx] / ref.sse_curve[ref.best_idx] - 1.0) <= 1e-6
        if idx == ref.best_idx:
            assert alpha == pytest.approx(ref.alpha, rel=1e-5) and sse == pytest.approx(ref.sse, rel=1e-5)


@pytest.mark.parametrize("s,k,bits1,bits2,signed,c1,c2,hf1,hf2,scale", [
    (4, 255, 4, 4, True, 16, 16, 1.0, 0.25, 1.0),       # one value fewer than the histogram path takes
    (5, 256, 4, 4, True, 16, 16, 1.0, 0.25, 1.0),
    (5, 257, 3, 5, True, 17, 5, 1.0, 1.0, 1.0),         # odd length, unequal bit widths, ratios up to 1
    (5, 1001, 2, 2, True, 32, 31, 0.7, 0.5, 1.0),
    (4, 900, 2, 6, False, 9, 16, 1.0, 0.3, 1.0),        # unsigned ranges: one side only
    (4, 900, 4, 4, False, 1, 1, 0.2, 0.1, 1.0),         # a single pair
    (3, 600, 4, 4, True, 12, 12, 3.0, 0.25, 1.0),       # scales beyond max|x|
    (3, 600, 4, 4, True, 8, 8, 1.0, 0.25, 2.0 ** -95),  # small values
    (2, 28672, 2, 3, True, 6, 6, 1.0, 0.25, 1.0),       # the longest row
    (3, 300, 4, 4, True, 3, 1024, 1.0, 0.9, 1.0),       # most ratios: sorted points of all of them in the workspace
    (3, 300, 2, 4, False, 2, 1024, 1.0, 1.0, 1.0),
    (3, 400, 4, 4, True, 4, 4, 1e-5, 0.25, 1.0),        # first scale far below max|x| ...
    (3, 400, 4, 4, True, 5, 5, 1e-7, 0.25, 1.0),        # ... and below its last place: equal errors take the lowest first code
    (3, 400, 3, 3, False, 5, 5, 1e-9, 0.5, 1.0),
])
def test_dual_search_by_bounds(s, k, bits1, bits2, signed, c1, c2, hf1, hf2, scale):
    import gpu_util
    from oracle import omse_oracle as orc
    t = synth.student_t3(s * k, seed=83, tensor_id=k).reshape(s, k) * np.float32(scale)
    alpha, sse, idx, q, pk = gpu_util.dual_quantize(t, bits1, bits2, signed, c1, c2, hf1, hf2, True, max(bits1, bits2) <= 4)
    ref = orc.dual_rows(t, bits1, bits2, signed, c1, c2, hf1, hf2)
    assert np.array_equal(idx, ref.best_idx) and np.array_equal(alpha, ref.alpha)
    np.testing.assert_allclose(sse, ref.sse, rtol=1e-5, atol=1e-37)
    assert np.array_equal(q.reshape(2, s, k), ref.codes)
    if pk is not None:
        for j in range(2):
            assert np.array_equal(pk[j], orc.pack_int4(ref.codes[j].reshape(-1)))


@pytest.mark.parametrize("s,k,bits,n_cand,hi_frac,scale", [
    (1300, 1, 4, 1024, 1.0, 1.0),                   # candidates evaluated, a warp per row: one value, one lane per candidate ...
    (1300, 27, 4, 1024, 1.0, 1.0), (1201, 63, 8, 200, 1.0, 1.0),
    (1201, 64, 3, 300, 1.0, 1.0), (1201, 65, 4, 1024, 1.0, 1.0),    # ... two lanes
    (1201, 127, 4, 1, 1.0, 1.0), (1201, 128, 4, 2, 1.0, 1.0),       # ... four; one and two candidates
    (1201, 160, 4, 4096, 1.0, 1.0), (1201, 161, 4, 4096, 1.0, 1.0), # one value more: by histogram
    (9, 27, 8, 1024, 1.0, 1.0), (9, 36, 4, 17, 0.3, 1.0), (9, 64, 4, 1024, 1.0, 1.0),     # small launches: 64 and 128 threads
    (9, 128, 4, 1024, 1.0, 1.0), (9, 129, 8, 1024, 1.0, 1.0),                             # ... the last row, by histogram
    (1201, 31, 4, 300, 1.0, 2.0 ** -112), (9, 40, 2, 300, 0.5, 2.0 ** 59),                # squares outside binary32
    (40, 700, 4, 4096, 0.1, 1.0), (40, 700, 8, 4096, 0.01, 2.0 ** -100),                  # by splits: bins do not fit
    (3, 12_287, 4, 4096, 0.1, 1.0), (3, 12_289, 4, 4096, 0.25, 1.0),                      # the last row by splits, windows
    (2, 25_600, 8, 4096, 0.05, 1.0), (2, 25_088, 4, 4096, 0.02, 1.0), (5, 5000, 4, 3, 1e-6, 1.0),
])
def test_residual_rows_by_every_search(s, k, bits, n_cand, hi_frac, scale):
    """Two quantized tensors, which rows of any length take through a block per row."""
    import gpu_util
    from oracle import omse_oracle as orc
    w = synth.student_t3(s * k, seed=101, tensor_id=k).reshape(s, k) * np.float32(scale)
    alpha, sse, q, pk = gpu_util.residual_quantize(w, (bits, bits), True, n_cand, hi_frac, 3, 1, True, bits <= 4)
    rows = np.unique(np.concatenate([np.arange(0, s, max(1, s // 40)), [s - 1]]))
    ref = orc.residual_rows(np.ascontiguousarray(w[rows]), (bits, bits), True, n_cand, hi_frac, 3, 1)
    # the two tensors of a row whose first scale differs by a rounding differ altogether: at most one row in fifty
    same = (alpha[0][rows] == ref.alpha[0]) & (alpha[1][rows] == ref.alpha[1])
    assert same.mean() >= 0.95 or (~same).sum() <= 1, same.mean()
    assert np.array_equal(q.reshape(2, s, k)[:, rows][:, same], ref.codes[:, same])
    np.testing.assert_allclose(sse[:, rows][:, same], ref.sse[:, same], rtol=1e-5, atol=1e-37)
    np.testing.assert_allclose(alpha[:, rows], ref.alpha, rtol=2e-2)
    if pk is not None:
        for j in range(2):
            assert np.array_equal(pk[j], orc.pack_int4(q[j]))


@pytest.mark.parametrize("bits1,bits2,signed,exponent", [
    (4, 4, True, -48), (4, 4, True, -56), (3, 4, False, -64), (4, 4, True, -68), (4, 4, True, -72), (2, 2, True, -76),    # squares below binary32
    (4, 4, True, 58), (4, 4, True, 62), (2, 4, False, 64), (4, 4, True, 66), (4, 4, True, 70),                            # ... and above
])
def test_dual_search_at_the_ends_of_binary32(bits1, bits2, signed, exponent):
    """The reference squares errors in binary32: equal squares take the lowest first code, infinite ones none."""
    import gpu_util
    from oracle import omse_oracle as orc
    t = synth.student_t3(3 * 600, seed=84, tensor_id=exponent % 97).reshape(3, 600) * np.float32(2.0 ** exponent)
    alpha, sse, idx, q, _ = gpu_util.dual_quantize(t, bits1, bits2, signed, 8, 8, 1.0, 0.25, True, False)
    ref = orc.dual_rows(t, bits1, bits2, signed, 8, 8, 1.0, 0.25)
    assert np.array_equal(idx, ref.best_idx) and np.array_equal(alpha, ref.alpha)
    assert np.array_equal(q.reshape(2, 3, 600), ref.codes)
    np.testing.assert_allclose(sse, ref.sse.astype(np.float32), rtol=1e-5, atol=1e-37)


@pytest.mark.parametrize("s,k,bits,signed,n_cand,hi_frac,kind", [
    (2101, 400, 4, True, 1024, 1.0, "student"),       # the shortest rows of that path, the finest fractions
    (1501, 1023, 4, True, 1024, 1.0, "extremes"),     # ten bits for the count, eleven from here on
    (1501, 1024, 4, False, 1000, 1.0, "student"),
    (1301, 1280, 5, True, 256, 1.0, "extremes"),
    (2401, 1281, 4, True, 500, 1.3, "student"),       # longer than a warp's registers hold; a grid beyond max|x|
    (2401, 2047, 8, True, 1024, 1.0, "extremes"),
    (2401, 2048, 4, True, 1024, 1.0, "extremes"),     # twelve bits for the count: the coarsest fractions
    (2371, 2304, 4, True, 1023, 1.0, "repeats"),      # a whole row in a few bins
    (2371, 2303, 8, False, 200, 1.0, "repeats"),
    (2101, 700, 8, True, 17, 1.0, "student"),         # fewer candidates than are looked at first
    (2101, 641, 4, True, 1024, 1.0, "scaled"),        # values that are scaled for their squares: a candidate per lane
    (2101, 640, 3, False, 1024, 1.0, "repeats"),
    (1301, 1280, 3, True, 1024, 1.0, "extremes"),     # fewer bits: by splits, and a block per row beyond
    (1301, 1281, 3, True, 1024, 1.0, "extremes"),
])
def test_rows_by_a_histogram_of_their_warp(s, k, bits, signed, n_cand, hi_frac, kind):
    import gpu_util
    w = synth.student_t3(s * k, seed=78, tensor_id=k).reshape(s, k)
    if kind == "extremes":                            # one value far above the others, of either sign: candidates all over the grid are open
        at = np.arange(0, s, 2)
        w[at, at % k] = np.where(at % 4 == 0, 1.0, -1.0).astype(np.float32) * np.float32(30.0) * (1.0 + at % 7).astype(np.float32)
    elif kind == "repeats":                           # all values on a lattice: thresholds meet them exactly
        w = np.clip(np.round(w * np.float32(2)), -9, 9).astype(np.float32) * np.float32(0.125)
        w[::5] = np.sign(w[::5]) * np.float32(0.25)   # one magnitude (and zeros)
    elif kind == "scaled":
        w = w * np.float32(2.0 ** 50)
    if not signed:
        w = np.abs(w)
    alpha, sse, idx, q, pk = gpu_util.quantize_weights(w, bits, signed, n_cand, hi_frac, 3, True, bits <= 4)
    rows = np.unique(np.concatenate([np.arange(0, s, 41), np.arange(0, s, 130), [s - 2, s - 1]]))
    st = check_rows(w, alpha, sse, idx, q, None, bits, signed, n_cand, hi_frac, 3, rows=rows)
    assert st["idx_diff"] <= max(1, st["rows"] // 50) and st["alpha_bitwise"] >= 0.99, st


@pytest.mark.parametrize("k,bits,n_cand", [(400, 4, 1024), (577, 4, 1024), (700, 5, 600), (703, 6, 1024), (1152, 6, 1024), (1152, 8, 1024),
                                           (1281, 8, 500), (2304, 4, 1024), (2304, 8, 1024)])
def test_unsigned_rows_of_both_signs_by_a_histogram(k, bits, n_cand):
    """Values of both signs on an unsigned range: a negative value errs by as much at every scale, however large it is, so it says
    nothing about the smallest scales.  Rows as they are drawn, with one large negative value, few positive ones, and none."""
    import gpu_util
    s = 1205
    w = synth.student_t3(s * k, seed=79, tensor_id=k).reshape(s, k)
    w[1::6, k // 2] = -8.0 * np.abs(w[1::6]).max(axis=1)
    w[2::6] = ((np.arange(k) % 97) / 97.0).astype(np.float32)              # a lattice of positive values beside one of -8
    w[2::6, 5] = -8.0
    w[3::6] = np.where(w[3::6] < 1.5, -np.abs(w[3::6]), w[3::6])
    w[4::6, ::2] = -2.0 * np.abs(w[4::6, ::2])
    w[::300] = -np.abs(w[::300])                                           # nothing to code: every scale is as good
    alpha, sse, idx, q, pk = gpu_util.quantize_weights(w, bits, False, n_cand, 1.0, 3, True, bits <= 4)
    rows = np.unique(np.concatenate([np.arange(0, s, 11), np.arange(0, s, 300), [s - 1]]))
    st = check_rows(w, alpha, sse, idx, q, None, bits, False, n_cand, 1.0, 3, rows=rows)
    assert st["idx_diff"] <= max(1, st["rows"] // 50) and st["alpha_bitwise"] >= 0.99, st


@pytest.mark.parametrize("shapes,bits,signed,launches", [
    ([(1801, 1280)], 3, True, 1), ([(1801, 1025)], 2, False, 1),       # all lanes and 40 values of a warp, in large numbers; by blocks otherwise
    ([(4801, 64), (297, 1153)], 3, True, 1),                           # beside many shorter rows, in one launch with them,
    ([(1501, 64), (21, 1152)], 4, True, 2),                            # by blocks beside fewer
    ([(1203, 1000), (21, 5000)], 4, True, 2),                          # few values by a histogram beside others: up to 1024 a row,
    ([(1101, 2304), (9, 5000)], 4, True, 1),                           # blocks beside blocks
    ([(303, 720), (4001, 128)], 8, False, 2), ([(61, 720), (4001, 128)], 8, True, 1),
    ([(38_001, 401)], 4, True, 1), ([(38_001, 449)], 4, True, 1), ([(38_001, 639)], 5, True, 1),
])
def test_rows_of_every_length_in_one_call(shapes, bits, signed, launches):
    """Lists on either side of the rules that give a tensor's rows to splits, to a histogram of their warp or to a block."""
    import torch
    import gpu_util
    ctx = gpu_util.ctx()
    ws = [synth.student_t3(s * k, seed=80, tensor_id=i).reshape(s, k) for i, (s, k) in enumerate(shapes)]
    descs = [dict(w=torch.from_numpy(w).cuda(), n_kernels=w.shape[0], kernel_len=w.shape[1], alpha=torch.empty(w.shape[0], device="cuda"),
                  sse=torch.empty(w.shape[0], device="cuda"), best_idx=torch.empty(w.shape[0], dtype=torch.int32, device="cuda"),
                  codes=torch.empty(w.size, dtype=torch.int8, device="cuda")) for w in ws]
    torch.cuda.synchronize()
    ctx.omse_read_launches()
    ctx.omse_quantize_weights_batched(descs, bits, signed, 300, 1.0, 3)
    assert ctx.omse_read_launches() == launches
    torch.cuda.synchronize()
    for w, d in zip(ws, descs):
        s = w.shape[0]
        rows = np.unique(np.concatenate([np.arange(0, s, max(1, s // 40)), [s - 1]]))
        st = check_rows(w, d["alpha"].cpu().numpy(), d["sse"].cpu().numpy(), d["best_idx"].cpu().numpy(), d["codes"].cpu().numpy(), None, bits,
                        signed, 300, 1.0, 3, rows=rows)
        assert st["idx_diff"] <= max(1, st["rows"] // 50) and st["alpha_bitwise"] >= 0.99, (w.shape, st)
