"""FP32 sums of high order over ranges of shifts: the powers of A must not leave
the range of FP32 where A itself is far inside it (N <= 12, and the shifts below
4096 of N = 13), nor the fourth powers of a state with a small norm.

Tolerance, u = 2^-24, squared norm n2: |dA| <= (N + 2) u n2; with a = 2 alpha, |d sum
|A|^a| <= a |dA| sum |A|^(a - 1) <= a (N + 2) u n2 d^(1/a) S^(1 - 1/a) (Hoelder), plus
the a + 16 roundings of powers and partial sums, (a + 16) u S."""
import numpy as np
import pytest

import oracle
from paper_2512_24685_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.fixture(scope="module")
def sre():
    import torch
    assert torch.cuda.is_available()
    from paper_2512_24685_gb300 import binding
    binding.load_library()
    return binding


def _tol(N, alpha, s, n2, shifts):
    a = 2 * alpha
    d = (1 << N) * shifts
    return a * (N + 2) * U * n2 * d ** (1 / a) * s ** (1 - 1 / a) + (a + 16) * U * s


# at the largest order of each size the largest |A|^(2 alpha) is about 2^-110
@pytest.mark.parametrize("N,alpha", [(4, 16), (8, 16), (10, 14), (10, 16), (11, 14), (12, 12), (12, 14), (12, 15), (13, 12), (16, 8)])
def test_ranges_without_the_first_shift(sre, N, alpha):
    import torch
    host = W.haar_state(N, 5 + N, np.complex64)
    d = min(1 << N, 4096)
    with sre.Plan(N, "c64") as p:
        for b, e in ((1, 9), (d - 7, d)):
            got = p.sum_pow_range(torch.from_numpy(host).cuda(), alpha, b, e)[0].item()
            ref = oracle.sum_pow_xorfwht(host, alpha, b, e)
            assert abs(got - ref) <= _tol(N, alpha, ref, 1.0, e - b), (b, got, ref)


@pytest.mark.parametrize("N", [6, 10])
def test_small_norms(sre, N):
    import torch
    scale = 2.0 ** -15  # squared norm 2^-30; A^4 down to 2^-140 at N = 10
    host = (scale * W.haar_state(N, 5 + N)).astype(np.complex64)
    n2 = float(np.sum(np.abs(host.astype(np.complex128)) ** 2))
    with sre.Plan(N, "c64") as p:
        got = p.sum4_range(torch.from_numpy(host).cuda(), 1, 1 << N)[0].item()
    ref = oracle.sum4_xorfwht(host, 1, 1 << N)
    # and half of FP32's smallest step per entry
    assert abs(got - ref) <= _tol(N, 2, ref, n2, 1 << N) + 2.0 ** (2 * N - 150), (got, ref)
