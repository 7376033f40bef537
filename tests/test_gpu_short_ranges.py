"""Ranges of a few hundred to 16383 shifts in the FP32 two-pass kernel: items of
two or four consecutive shifts.  A shift's sum does not depend on the shifts that
it shares an item with, so per-shift sums equal those of very short ranges (one
shift per item) bit for bit."""
import numpy as np
import pytest

from paper_2512_24685_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sre():
    import torch
    assert torch.cuda.is_available()
    from paper_2512_24685_gb300 import binding
    binding.load_library()
    return binding


# N = 20: below 4096 the shifts beside the tensor-core kernel
@pytest.mark.parametrize("N,mode,ranges", [
    (17, "fp32", [(0, 256), (4095, 4095 + 1023), (8190, 8190 + 1024), (60001, 60001 + 16383)]),
    (18, "fp32", [(0, 1025), (8191, 8191 + 259), ((1 << 18) - 5003, 1 << 18)]),
    (19, "fp32", [(1, 1026), (262143, 262143 + 301)]),
    (20, "fp16_split", [(0, 1030), (3801, 4096)])])
def test_per_shift_sums_do_not_depend_on_the_range(sre, N, mode, ranges):
    import torch
    psi = torch.from_numpy(W.haar_state(N, 3 + N, np.complex64)).cuda()
    with sre.Plan(N, "c64", mode) as p:
        for b, e in ranges:
            out, px = p.sum4_range(psi, b, e, per_x=True)
            for a in (b, (b + e) // 2, e - 9):
                _, py = p.sum4_range(psi, a, a + 9, per_x=True)
                assert torch.equal(px[a - b:a - b + 9], py), (b, e, a)
            assert abs(out[0].item() - px.sum().item()) <= 1e-13 * out[0].item()


@pytest.mark.parametrize("alpha", [3, 6])
def test_orders_in_short_ranges(sre, alpha):
    import torch
    psi = torch.from_numpy(W.haar_state(17, 3, np.complex64)).cuda()
    with sre.Plan(17, "c64") as p:
        _, px = p.sum_pow_range(psi, alpha, 8185, 8185 + 300, per_x=True)
        _, py = p.sum_pow_range(psi, alpha, 8185, 8185 + 20, per_x=True)
    assert torch.equal(px[:20], py)


def _us(call, reps=200):
    import torch
    best = float("inf")
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            call()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b) / reps * 1e3)
    return best


def test_one_shift_of_a_small_state_costs_no_more_than_many(sre):
    """The norm of a state in one tile is spread over CTAs however short the
    range is (by the range's only CTA: 35 us against 21).  30 % between runs."""
    import torch
    psi = torch.from_numpy(W.haar_state(12, 3, np.complex64)).cuda()
    with sre.Plan(12, "c64") as p:
        n2 = [p.sum4_range(psi, b, e)[1].item() for b, e in ((0, 4096), (5, 6), (4000, 4003), (0, 70))]
        assert len(set(n2)) == 1
        assert _us(lambda: p.sum4_range(psi, 5, 6)) <= 1.3 * _us(lambda: p.sum4_range(psi, 0, 64))


def test_a_handful_of_shifts_in_a_split_mode_takes_small_items(sre):
    """One shift of N = 18 beside the same with an L2-sized ring of small chunks,
    which a caller can ask for (in chunks of eight shifts 24 % slower).  10 %
    between runs."""
    import torch
    psi = torch.from_numpy(W.haar_state(18, 3, np.complex64)).cuda()
    x = (1 << 17) + 1
    with sre.Plan(18, "c64", "fp16_split") as p:
        library = _us(lambda: p.sum4_range(psi, x, x + 1))
        p.set_tuning(1, 23, 11, 3, 0)
        assert library <= 1.1 * _us(lambda: p.sum4_range(psi, x, x + 1))
