"""Values on a lattice of their own: equal values in large numbers, at or within a few units in the last place of the
thresholds of the search grid.  There a value counted on the wrong side of a threshold moves the error of a candidate by far more
than among values drawn from a density."""
import numpy as np
import pytest

from paper_1902_06822_b200 import synth

pytestmark = pytest.mark.gpu


def _repeat(*pairs):
    return np.concatenate([np.full(n, v, np.float32) for v, n in pairs])


def _ulps(v, n):
    return (np.float32(v).view(np.int32) + np.int32(n)).view(np.float32)


def _beside_edges(n, n_cand, most, seed):
    """Odd multiples of half a grid step below `most`, up to two units in the last place away; and `most` itself."""
    rng = np.random.default_rng(seed)
    h = np.float32(np.float32(most) / np.float32(n_cand)) * np.float32(0.5)
    x = ((2 * rng.integers(0, n_cand, n) + 1) * h.astype(np.float64)).astype(np.float32)
    x = (x.view(np.int32) + rng.integers(-2, 3, n).astype(np.int32)).view(np.float32)
    x = np.minimum(x, np.float32(most))
    x[n // 2] = most
    return x


def _bytes(n, scale, seed):
    return (np.random.default_rng(seed).integers(0, 256, n).astype(np.float32) * np.float32(scale)).astype(np.float32)


def _signs(x, seed):
    return np.where(np.random.default_rng(seed).random(x.size) < 0.5, -x, x).astype(np.float32)


# one value under each of these shapes errs by 1e-5 of the smallest error or more when it is put on the wrong side
TENSORS = [
    ("ties_at_the_best", lambda: _repeat((0.945, 174), (0.5250001, 61), (0.87500006, 4), (0.275, 155), (0.88, 141), (1.0, 1)), 8, False, 100),
    ("one_value_above_an_edge", lambda: _repeat((_ulps(771 / 1024, 2), 20000), (1.0, 1)), 8, False, 512),
    ("one_value_below_an_edge", lambda: _repeat((_ulps(771 / 1024, -2), 20000), (1.0, 1)), 8, False, 512),
    ("multiples_of_0.05", lambda: np.round(np.abs(synth.student_t3(20001, seed=91)) * np.float32(20)) * np.float32(0.05), 8, False, 500),
    ("multiples_of_0.05_signed", lambda: np.round(synth.student_t3(20001, seed=92) * np.float32(20)) * np.float32(0.05), 4, True, 500),
    ("bytes", lambda: _bytes(30_003, 0.0123, 93), 4, False, 1000),
    ("bytes_8", lambda: _bytes(30_003, 1 / 255, 94), 8, False, 500),
    ("beside_edges", lambda: _beside_edges(9001, 777, 1.0, 95), 8, False, 777),
    ("beside_edges_signed", lambda: _signs(_beside_edges(9001, 1000, 0.37, 96), 97), 8, True, 1000),
    ("beside_edges_4", lambda: _signs(_beside_edges(9001, 500, 3.1, 98), 99), 4, True, 500),
]


@pytest.mark.parametrize("path", ["context", "static", "grid_below"])
@pytest.mark.parametrize("case", range(len(TENSORS)), ids=[t[0] for t in TENSORS])
def test_per_tensor_search_on_lattice_values(case, path):
    """In one kernel, through the pipeline, and with a grid that ends below max|x| (values above the last threshold, windows)."""
    import torch

    import gpu_util
    from oracle import omse_oracle as orc
    from paper_1902_06822_b200 import binding
    _, make, bits, signed, n_cand = TENSORS[case]
    x, hi_frac = make().astype(np.float32), 1.0
    if path == "grid_below":          # one value 50 times as large: the same steps, and with them the same ties
        x, hi_frac = np.concatenate([x, np.float32([50]) * np.abs(x).max()]), 0.02
    if path == "static":
        d_x = torch.from_numpy(x).cuda()
        out, idx = torch.zeros(2, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        curve = torch.zeros(n_cand, dtype=torch.float64, device="cuda")
        binding.omse_activation_scale_static(d_x, x.size, bits, signed, n_cand, hi_frac, 3, out[:1], out[1:], idx, curve)
        alpha, sse, idx, curve = out[0].item(), out[1].item(), idx.item(), curve.cpu().numpy()
    else:
        alpha, sse, idx, curve = gpu_util.activation_scale(x, bits, signed, n_cand, hi_frac, 3)
    ref = orc.activation_scale(x, bits, signed, n_cand, hi_frac, 3)
    assert idx >= 0
    assert ref.sse_curve[idx] - ref.sse_curve[ref.best_idx] <= 1e-6 * ref.sse_curve[ref.best_idx], (idx, ref.best_idx)
    # A value within 2^-23 of a threshold may be coded to either neighbour (the scale's rounding, the quotient's): its error
    # then moves by 2*alpha times its distance from the midpoint.  Everything else is summed in binary64.
    m = np.float32(np.float32(hi_frac) * np.abs(x).max())
    step = np.float32(m / np.float32(n_cand))
    scales = (np.arange(1, n_cand + 1, dtype=np.float32) * step).astype(np.float64)
    t = np.abs(x.astype(np.float64))[None, :] / scales[:, None]
    beside = np.abs(t - (np.floor(t) + 0.5)) <= 1.25e-7 * t
    slack = 2.5e-7 * scales * (beside * np.abs(x.astype(np.float64))).sum(axis=1)
    ok = ref.sse_curve > 1e-8 * (x.astype(np.float64) ** 2).sum()
    assert np.all(np.abs(curve - ref.sse_curve)[ok] <= (2e-6 * ref.sse_curve + slack)[ok])
    if idx != ref.best_idx:
        ref = orc.phi(x, bits, signed, n_cand, hi_frac, 3, start_idx=idx, want_codes=False)
    assert alpha == pytest.approx(ref.alpha, rel=1e-5, abs=0)
    assert sse == pytest.approx(ref.sse, rel=1e-5, abs=1e-37)


@pytest.mark.parametrize("hi_frac", [1.0, 0.03])           # all bins at once; bins in windows, values above the last threshold
@pytest.mark.parametrize("case", range(len(TENSORS)), ids=[t[0] for t in TENSORS])
def test_rows_on_lattice_values(case, hi_frac):
    import gpu_util
    from parity import check_rows
    _, make, bits, signed, n_cand = TENSORS[case]
    x = make().astype(np.float32)
    n_cand = n_cand if hi_frac == 1.0 else 4000
    w = np.resize(np.random.default_rng(5).permutation(x), (3, 900))
    w[:, 0] = np.abs(x).max() / np.float32(hi_frac)
    alpha, sse, idx, q, _ = gpu_util.quantize_weights(w, bits, signed, n_cand, hi_frac, 3, True, False)
    check_rows(w, alpha, sse, idx, q, None, bits, signed, n_cand, hi_frac, 3)
