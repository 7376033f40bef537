"""Tunings of the FP32 two-pass kernels that were saved for other kernels.  N =
17..19 take none: a saved one changes neither the order of the sums (bit for
bit) nor the share of the work that is done twice."""
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


@pytest.mark.parametrize("N,tuning", [(17, (2, 55, 27, 3, 0, 1, 1)), (17, (0, 9, 4, 1, 1, 0, 0)),
                                      (18, (3, 23, 11, 3, 0, 1, 1)), (19, (0, 40, 20, 3, 1, 1, 1))])
def test_saved_tunings_leave_the_kernel_as_it_is(sre, N, tuning):
    import numpy as np
    import torch
    psi = torch.from_numpy(W.haar_state(N, 9 + N, np.complex64)).cuda()
    with sre.Plan(N, "c64") as p:
        for b, e in ((5, 5 + 40001), (8192, 8192 + 300)):
            want = p.sum4_range(psi, b, e).tolist()
            p.set_tuning(*tuning)
            got = p.sum4_range(psi, b, e).tolist()
            p.set_tuning(-1, -1, -1, -1, -1)
            assert got == want
        p.set_tuning(3, 64, 5)  # a ring beyond the plan's scratch is refused as ever
        with pytest.raises(sre.SreError):
            p.sum4_range(psi, 0, 8)


def test_twenty_qubits_take_the_tuned_kernel(sre):
    """N = 20: the general two-pass kernel, which a saved tuning was found for;
    with it a range takes no longer than with the library's choice (10 % between
    runs; read by the item-list kernel it took 43 % longer)."""
    import numpy as np
    import torch
    psi = torch.from_numpy(W.haar_state(20, 29, np.complex64)).cuda()
    b, n = 8192 + 77, 32768

    def ms(p):
        p.set_profiling(True)
        p.sum4_range(psi, b, b + n)
        runs = []
        for _ in range(3):
            p.sum4_range(psi, b, b + n)
            t, name = p.last_kernel_ms()
            assert name == "k_large"
            runs.append(t)
        return min(runs)

    with sre.Plan(20, "c64") as p:
        library = ms(p)
        p.set_tuning(0, 47, 23, 3, 3, 1, 1)
        assert ms(p) <= 1.1 * library


def test_twenty_qubits_alike_for_every_range_and_server(sre):
    """N = 20: a shift's sum does not depend on the length of its range, nor M2 on
    whether a plan or a server with a shorter ring forms it (range sums add the
    same doubles in another order: n 2^-52)."""
    import numpy as np
    import torch
    host = W.haar_state(20, 29, np.complex64)
    psi = torch.from_numpy(host).cuda()
    with sre.Plan(20, "c64") as p:
        _, px = p.sum4_range(psi, 4090, 4090 + 200, per_x=True)
        for a, n in ((4090, 1), (4095, 3), (4200, 15), (4100, 64)):
            _, py = p.sum4_range(psi, a, a + n, per_x=True)
            assert torch.allclose(px[a - 4090:a - 4090 + n], py, rtol=2.0 ** -48, atol=0)
        want = p.m2(psi)
    with sre.Server(max_inflight=1, max_N=20) as srv:
        assert abs(srv.wait(srv.submit(host), 120000) - want) <= 2.0 ** (20 - 52)
