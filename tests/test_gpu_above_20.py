"""Sizes above 20 qubits, where the general two-pass kernel runs every shift
itself: FP32 with the pivot inside a block, x = 0 and pass-2 tiles by tensor copy
(N = 21), fixed point with pass 2 over eight bits (N = 21) and over more, on one
move buffer (N = 22).

Tolerances of a per-shift sum.  FP32, u = 2^-24: as for the smaller sizes, |dA|
<= (N + 2) u (squared norm 1), so 4 (N + 2) u d^(1/4) S^(3/4) by Hoelder, plus 16
u S for the partial sums.  FP64, u = 2^-53 and G = sum_t |g_x(t)|: |dA| <= (N + 27) u
G for the oracle's butterflies and the fixed point together, so 4 (N + 27) u G
d^(1/4) S^(3/4), plus 2^-50 S."""
import numpy as np
import pytest

import oracle
from paper_2512_24685_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sre():
    import torch
    assert torch.cuda.is_available()
    from paper_2512_24685_gb300 import binding
    binding.load_library()
    return binding


def _state(N, family):
    return W.haar_state(N, 31 + N) if family == "haar" else W.product_state(N, 57 + N)[0]


def _ranges(N):
    d = 1 << N
    return (0, 3), (4094, 4098), (d // 2 - 1, d // 2 + 1), (d - 2, d)


# one shift per chunk takes the block pairs by bulk copy, eight share the loads
@pytest.mark.parametrize("tuning", [(), (0, 9, 4, 2, 1), (3, 3, 1, 2, 0), (0, 9, 4, 2, 1, 0, 0)])
@pytest.mark.parametrize("family", ["haar", "product"])
def test_fp32_per_shift_sums(sre, family, tuning):
    import torch
    N = 21
    host = _state(N, family).astype(np.complex64)
    psi = torch.from_numpy(host).cuda()
    with sre.Plan(N, "c64") as p:
        if tuning:
            p.set_tuning(*tuning)
        for b, e in _ranges(N):
            out, px = p.sum4_range(psi, b, e, per_x=True)
            got = px.cpu().numpy()
            assert abs(out[0].item() - got.sum()) <= 1e-14 * got.sum()
            for k, x in enumerate(range(b, e)):
                ref = oracle.sum4_xorfwht(host, x, x + 1)
                tol = 4 * (N + 2) * 2.0 ** -24 * 2 ** (N / 4) * ref ** 0.75 + 2.0 ** -20 * ref
                assert abs(got[k] - ref) <= tol, (x, got[k], ref)


@pytest.mark.parametrize("family", ["haar", "product"])
@pytest.mark.parametrize("N", [21, 22])
def test_fp64_per_shift_sums(sre, N, family):
    import torch
    host, d = _state(N, family), 1 << N
    psi, t = torch.from_numpy(host).cuda(), np.arange(d)
    with sre.Plan(N, "c128", "fp64") as p:
        for b, e in _ranges(N):
            out, px = p.sum4_range(psi, b, e, per_x=True)
            got = px.cpu().numpy()
            assert abs(out[0].item() - got.sum()) <= 1e-14 * got.sum()
            for k, x in enumerate(range(b, e)):
                ref = oracle.sum4_xorfwht(host, x, x + 1)
                g = float(np.sum(np.abs(host) * np.abs(host[t ^ x])))
                tol = 4 * (N + 27) * 2.0 ** -53 * g * 2 ** (N / 4) * ref ** 0.75 + 2.0 ** -50 * ref
                assert abs(got[k] - ref) <= tol, (x, got[k], ref)
