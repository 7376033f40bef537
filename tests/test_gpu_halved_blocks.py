"""The FP32 block kernels (N = 13..16 in one pass, N = 17..20 in two): every
shift runs halved, so the sizes where they can go wrong are the shifts whose
pivot lies inside a block (x < 8192), x = 0, the first shift with the pivot
above it, ragged ranges and odd counts, and states at an 8-byte offset.

Tolerance of a per-shift sum: with u = 2^-24 and the N + 2 roundings of a
product and its transform, |dA| <= (N + 2) u sum_t |g_x(t)| <= (N + 2) u (n2 = 1);
then |d sum A^4| <= 4 max|dA| sum |A|^3 <= 4 (N + 2) u d^(1/4) S_x^(3/4) (Hoelder),
plus 16 roundings of the FP32 partial sums, 16 u S_x.  The shift x = 0 at order
alpha scales the first term by alpha / 2 with S_x the order-alpha sum's bound."""
import numpy as np
import pytest

import oracle
from paper_2512_24685_gb300 import workloads as W

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


def tol(N, s):
    return 4 * (N + 2) * U * 2 ** (N / 4) * s ** 0.75 + 16 * U * s


@pytest.fixture(scope="module")
def sre():
    import torch
    assert torch.cuda.is_available()
    from paper_2512_24685_gb300 import binding
    binding.load_library()
    return binding


def _state(N, family):
    return W.haar_state(N, 31 + N, np.complex64) if family == "haar" else W.product_state(N, 57 + N, np.complex64)[0]


@pytest.mark.parametrize("family", ["haar", "product"])
@pytest.mark.parametrize("N", [13, 14, 15, 16, 17, 18, 19, 20])
def test_per_shift_sums_at_the_edges(sre, N, family):
    import torch
    host = _state(N, family)
    psi = torch.from_numpy(host).cuda()
    off = torch.zeros((1 << N) + 1, dtype=torch.complex64, device="cuda")
    off[1:] = psi
    d = 1 << N
    ranges = [(0, 9), (4094, 4099), (8190, min(d, 8195)), (d // 2 - 1, d // 2 + 2), (d - 3, d)]
    with sre.Plan(N, "c64") as p:
        for b, e in ranges:
            if b >= e:
                continue
            out, px = p.sum4_range(psi, b, e, per_x=True)
            _, py = p.sum4_range(off[1:], b, e, per_x=True)
            got = px.cpu().numpy()
            assert torch.equal(px, py)
            assert abs(out[0].item() - got.sum()) <= 1e-14 * got.sum()
            for k, x in enumerate(range(b, e)):
                ref = oracle.sum4_xorfwht(host, x, x + 1)
                assert abs(got[k] - ref) <= tol(N, ref), (N, x, got[k], ref)


@pytest.mark.parametrize("N,tuning", [(17, ()), (18, (0, 3, 1)), (18, (1, 64, 5)), (18, (3, 4, 1)), (19, (2, 5, 2))])
def test_ragged_ranges_share_no_shift_twice(sre, N, tuning):
    """Ranges long enough for shared factor loads (16384 shifts and more),
    ragged at both ends: the same per-shift sums as short ranges give."""
    import torch
    psi = torch.from_numpy(_state(N, "haar")).cuda()
    b, n = 8192 + 77, 16384 + 1001
    with sre.Plan(N, "c64") as p:
        if tuning:
            p.set_tuning(*tuning)
        out, px = p.sum4_range(psi, b, b + n, per_x=True)
        for a in (b, b + 8111, b + n - 64):
            _, py = p.sum4_range(psi, a, a + 64, per_x=True)
            assert torch.equal(px[a - b:a - b + 64], py)
        assert abs(out[0].item() - px.sum().item()) <= 1e-13 * out[0].item()


@pytest.mark.parametrize("alpha", [3, 5])
@pytest.mark.parametrize("N", [13, 15, 16, 17])
def test_order_alpha_sums(sre, N, alpha):
    import torch
    host = _state(N, "product")
    psi = torch.from_numpy(host).cuda()
    with sre.Plan(N, "c64") as p:
        _, px = p.sum_pow_range(psi, alpha, 0, 5, per_x=True)
    for x in range(5):
        ref = oracle.sum_pow_xorfwht(host, alpha, x, x + 1)
        # |A| <= 1: the order-alpha derivative is at most 2 alpha |A|^3
        s4 = oracle.sum4_xorfwht(host, x, x + 1)
        assert abs(px[x].item() - ref) <= alpha / 2 * tol(N, s4)


def test_batch_of_every_block_size_equals_single(sre):
    import torch
    Ns = [16, 13, 17, 14, 15, 13, 18, 16]
    states = [torch.from_numpy(_state(n, "haar" if k % 2 else "product")).cuda() for k, n in enumerate(Ns)]
    with sre.Plan(18, "c64") as p:
        got = p.m2_batched(states).tolist()
        assert got == [p.m2(s) for s in states]
