"""Per-shift sums of the FP64 mode where the large entries of the two factors of
g_x do not meet, so that the products lie many orders of magnitude below the
block norms: states close to a basis state, shifts of high weight.

Tolerance, u = 2^-53 and G = sum_t |g_x(t)| (halved form): the oracle's FP64
butterflies keep |dA| <= (N + 4) u G.  Fixed point: 2 u G from the products, 16
u G from their quantization (half of 2^-60 of a block's largest product, 4096
times), 5 u G from the rescaling between groups of stages.  With |dA| <= D =
(N + 27) u G, Hoelder gives |d sum A^4| <= 4 D d^(1/4) S^(3/4); the sums of powers
add 2^-50 S."""
import numpy as np
import pytest

import oracle
from paper_2512_24685_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def sre():
    import torch
    assert torch.cuda.is_available()
    from paper_2512_24685_gb300 import binding
    binding.load_library()
    return binding


def _near_basis(N, angle, phases):
    r = np.random.default_rng(N)
    psi = np.ones(1, np.complex128)
    for _ in range(N):
        one = np.sin(angle / 2) * (np.exp(2j * np.pi * r.random()) if phases else 1.0)
        psi = np.concatenate([psi * np.cos(angle / 2), psi * one])
    return psi


def _state(N, kind):
    if kind == "basis+haar":
        psi = 1e-6 * W.haar_state(N, 5 + N)
        psi[0] += 1
        return psi / np.linalg.norm(psi)
    return _near_basis(N, *{"0.2": (0.2, True), "0.1": (0.1, True), "0.01": (0.01, True), "0.1 real": (0.1, False),
                            "0.01 real": (0.01, False)}[kind])


def _check(N, psi, x, got):
    d = 1 << N
    ref = oracle.sum4_xorfwht(psi, x, x + 1)
    g = float(np.sum(np.abs(psi) * np.abs(psi[np.arange(d) ^ x])))
    tol = 4 * (N + 27) * U * g * d ** 0.25 * ref ** 0.75 + 2.0 ** -50 * ref
    assert abs(got - ref) <= tol, (N, x, got, ref, tol)


@pytest.mark.parametrize("kind", ["0.2", "0.1", "0.01", "0.1 real", "0.01 real", "basis+haar"])
@pytest.mark.parametrize("N", [2, 5, 8, 9, 10, 12, 13, 14, 15, 16, 17, 18])
def test_per_shift_sums_scale_with_the_products(sre, N, kind):
    import torch
    psi = _state(N, kind)
    t, d = torch.from_numpy(psi).cuda(), 1 << N
    with sre.Plan(N, "c128", "fp64") as p:
        for x in sorted({0, 1, d // 2, d - 1 - d // 16, d - 2, d - 1}):
            if N <= 12:
                _check(N, psi, x, p.sum4_range(t, x, x + 1)[0].item())
            else:
                out, px = p.sum4_range(t, x, x + 1, per_x=True)
                assert px[0].item() == out[0].item()
                _check(N, psi, x, px[0].item())
