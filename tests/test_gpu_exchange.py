"""The exchanges between the blocks of the one-kernel per-tensor search."""
import numpy as np
import pytest

from paper_1902_06822_b200 import synth

pytestmark = pytest.mark.gpu


def _outputs(n_cand):
    import torch
    return (torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"),
            torch.zeros(n_cand, dtype=torch.float64, device="cuda"))


@pytest.mark.parametrize("n,bits,n_cand", [(1_605_633, 8, 500), (303_105, 4, 1024), (25_088, 4, 50)])
def test_repeated_searches_give_the_same_bits(n, bits, n_cand):
    """Every block sees all additions to the histogram and all re-scored errors: calls in a row on two tensors in turn."""
    import torch

    import gpu_util
    from oracle import omse_oracle as orc
    xs = [np.abs(synth.student_t3(n, seed=61 + i)) for i in range(2)]
    xs[1] = np.round(xs[1] * np.float32(8)) * np.float32(0.125)        # many candidates to re-score
    d_xs = [torch.from_numpy(x).cuda() for x in xs]
    first = []
    for rep in range(150):
        for i, d_x in enumerate(d_xs):
            out = _outputs(n_cand)
            gpu_util.ctx().omse_activation_scale(d_x, n, bits, False, n_cand, 1.0, 3, *out)
            if rep == 0:
                first.append(out)
            else:
                assert all(torch.equal(a, b) for a, b in zip(out, first[i])), (rep, i)
    for x, out in zip(xs, first):
        ref = orc.activation_scale(x, bits, False, n_cand, 1.0, 3)
        assert out[0].item() == pytest.approx(ref.alpha, rel=1e-5) and out[1].item() == pytest.approx(ref.sse, rel=1e-5)


@pytest.mark.parametrize("n", [303_105, 25_088, 100])
def test_a_wait_that_runs_out_is_reported_and_leaves_no_trace(n):
    """With few polls allowed (or none) blocks give up: the status says so, and calls before and after are not affected."""
    import torch

    from paper_1902_06822_b200 import binding
    ctx = binding.Context(0)
    d_x = torch.from_numpy(np.abs(synth.student_t3(n, seed=65))).cuda()

    def search():
        out = _outputs(300)
        ctx.omse_activation_scale(d_x, n, 4, False, 300, 1.0, 3, *out)
        return out, ctx.omse_last_device_status()

    good, status = search()
    assert status == 0
    for polls in [0, 1, 2, 3, 4, 8, 16, 32, 64] * 3:
        ctx.omse_set_poll_limit(polls)
        out, status = search()
        if polls == 0:
            assert status & binding.DEV_INCOMPLETE
        if not status & binding.DEV_INCOMPLETE:        # nobody gave up: the result is whole
            assert status == 0 and all(torch.equal(a, b) for a, b in zip(out, good))
        ctx.omse_set_poll_limit(1 << 22)
        out, status = search()
        assert status == 0 and all(torch.equal(a, b) for a, b in zip(out, good)), polls
    ctx.close()


def test_a_refused_launch_takes_the_sequence_of_launches():
    """More blocks than the GPU runs at once (each takes most of an SM's shared memory): the driver refuses, the call does not."""
    import torch

    from oracle import omse_oracle as orc
    from paper_1902_06822_b200 import binding
    n = 160 * 40_000                                    # 160 KB of values per block
    if torch.cuda.get_device_properties(0).multi_processor_count >= 160:
        pytest.skip("as many SMs as the search has blocks at most")
    ctx = binding.Context(0)
    x = np.abs(synth.student_t3(n, seed=66))
    d_x = torch.from_numpy(x).cuda()
    ctx.omse_set_search_blocks(160)
    out = _outputs(100)
    ctx.omse_read_launches()
    ctx.omse_activation_scale(d_x, n, 4, False, 100, 1.0, 3, *out)
    assert ctx.omse_last_device_status() == 0
    assert ctx.omse_read_launches() > 5                 # not in one kernel
    ref = orc.activation_scale(x, 4, False, 100, 1.0, 3)
    assert out[2].item() == ref.best_idx and out[0].item() == pytest.approx(ref.alpha, rel=1e-5)
    assert out[1].item() == pytest.approx(ref.sse, rel=1e-5)
    # nothing of the refusal is left for the next call, whatever its path
    w = torch.from_numpy(synth.student_t3(64 * 300, seed=67)).cuda()
    a, s = torch.zeros(64, device="cuda"), torch.zeros(64, device="cuda")
    ctx.omse_quantize_weights(w, 64, 300, 4, True, 100, 1.0, 3, a, s)
    ctx.omse_set_search_blocks(20)                      # fewer blocks than SMs: in one kernel again
    small = _outputs(100)
    ctx.omse_activation_scale(d_x, 303_105, 4, False, 100, 1.0, 3, *small)
    assert ctx.omse_last_device_status() == 0 and ctx.omse_read_launches() == 2
    ref = orc.activation_scale(x[:303_105], 4, False, 100, 1.0, 3)
    assert small[2].item() == ref.best_idx and small[0].item() == pytest.approx(ref.alpha, rel=1e-5)
    ctx.close()
