"""The tensor-core kernel's library ring (N = 16..20 in the split modes) and
what completes a caller's partial tuning.  A shift's sum does not depend on how
shifts share chunks and slots, so per-shift sums are compared bit for bit; the
range sum adds the same n doubles in another order: relative error <= n 2^-52."""
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


@pytest.mark.parametrize("N,mode", [(16, "fp16_split"), (17, "bf16_split"), (18, "fp16_split"), (19, "bf16_split"),
                                    (20, "fp16_split")])
def test_library_ring_gives_the_sums_of_a_small_ring(sre, N, mode):
    import torch
    psi = torch.from_numpy(W.haar_state(N, 5 + N, np.complex64)).cuda()
    g2 = min(5, N - 13)
    b, n = 4096 + 3, 2048 + 5
    with sre.Plan(N, "c64", mode) as p:
        out, px = p.sum4_range(psi, b, b + n, per_x=True)
        p.set_tuning(0, 9, 4, g2, 0)
        o1, p1 = p.sum4_range(psi, b, b + n, per_x=True)
    assert torch.equal(px, p1)
    assert abs(out[0].item() - o1[0].item()) <= n * 2.0 ** -52 * o1[0].item()


@pytest.mark.parametrize("N,mode", [(16, "fp16_split"), (17, "fp16_split"), (18, "fp32"), (20, "fp32"), (20, "fp16_split")])
def test_partial_tunings_are_taken(sre, N, mode):
    """Each ring field alone, at the ends of what the L2-sized ring allows."""
    import torch
    psi = torch.from_numpy(W.haar_state(N, 5 + N, np.complex64)).cuda()
    b, n = 4096 + 3, 61
    with sre.Plan(N, "c64", mode) as p:
        want = p.sum4_range(psi, b, b + n)[0].item()
        lag, ring = {16: (31, 63), 17: (20, 41), 18: (11, 23), 20: (4, 9)}[N]
        for t in ({"x_batch_log": 0}, {"ring_slots": lag + 1}, {"ring_slots": ring}, {"lag": 1}, {"lag": ring - 1}):
            p.set_tuning(**t)
            got = p.sum4_range(psi, b, b + n)[0].item()
            # a lane adds 16 + at most 32 FP32 terms per item, grouped by the
            # item's size: 64 roundings of 2^-24 on each side
            assert abs(got - want) <= 2.0 ** -17 * want, t


@pytest.mark.parametrize("mode", ["fp32", "fp16_split"])
def test_a_plan_s_library_tuning_serves_a_server(sre, mode):
    import torch
    v = W.haar_state(18, 44, np.complex64)
    with sre.Plan(18, "c64", mode) as p:
        want, t = p.m2(torch.from_numpy(v).cuda()), p.get_tuning(18)
    with sre.Server(max_inflight=1, max_N=18, mode=mode, slot_scratch_bytes=96 << 20) as srv:
        srv.set_tuning(18, t)
        # log2 of a sum whose 2^18 terms are added in another order
        assert abs(srv.wait(srv.submit(v)) - want) <= 2 * 2.0 ** (18 - 52)
