"""The FP64 mode's fixed-point transform at the states where a unit could be
too coarse or overflow: amplitudes spread over many orders of magnitude, blocks
of zeros, a basis state, norms far from one, x = 0 and pivots inside a block.

Tolerance of a per-shift sum: the FP64 oracle and the fixed-point transform
each carry at most u = 2^-53 per rounding of the partial sums, N + 4 of them, of
a value bounded by G = sum_t |g_x(t)| (and 2^-50 of the block pairs' bounds, which
sum to B >= G): |dA| <= 2 (N + 4) u B, so |d sum A^4| <= 8 (N + 4) u B d^(1/4)
S_x^(3/4) (Hoelder), plus the sum's own 2^-50 S_x."""
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


def _state(N, kind):
    d = 1 << N
    if kind == "haar":
        return W.haar_state(N, 11 + N)
    if kind == "product":
        return W.product_state(N, 13 + N)[0]
    if kind == "stabilizer":
        return W.stabilizer_state(N, 17 + N, depth=8)
    if kind == "basis":
        return W.basis_state(N, d // 3)
    v = W.haar_state(N, 19 + N) * 10.0 ** (-9.0 * np.arange(d) / d)
    if kind == "gaps":  # blocks of 4096 zeros, or zero runs in a small state
        v.reshape(-1, max(1, min(4096, d // 4)))[1::2] = 0
    return v / np.linalg.norm(v)


def _bound(psi, x, N):
    """Sum over the block pairs of the product of their l2 norms."""
    if N <= 12 or x < 4096:
        return float(np.sum(np.abs(psi) ** 2))
    n = np.sqrt(np.sum(np.abs(psi.reshape(-1, 4096)) ** 2, axis=1))
    return float(np.sum(n * n[np.arange(n.size) ^ (x >> 12)])) / 2


@pytest.mark.parametrize("kind", ["haar", "product", "stabilizer", "basis", "decay", "gaps"])
@pytest.mark.parametrize("N", [13, 14, 15, 16])
def test_per_shift_sums(sre, N, kind):
    import torch
    psi = _state(N, kind)
    t, d = torch.from_numpy(psi).cuda(), 1 << N
    with sre.Plan(N, "c128", "fp64") as p:
        for b, e in ((0, 4), (4094, 4098), (d // 2 - 1, d // 2 + 1), (d - 2, d)):
            out, px = p.sum4_range(t, b, e, per_x=True)
            got = px.cpu().numpy()
            assert abs(out[0].item() - got.sum()) <= 2.0 ** -48 * got.sum()
            for k, x in enumerate(range(b, e)):
                ref = oracle.sum4_xorfwht(psi, x, x + 1)
                tol = 8 * (N + 4) * U * _bound(psi, x, N) * 2 ** (N / 4) * ref ** 0.75 + 2.0 ** -50 * ref
                assert abs(got[k] - ref) <= tol + 1e-300, (N, kind, x, got[k], ref)


@pytest.mark.parametrize("kind", ["haar", "stabilizer", "basis", "decay", "gaps"])
@pytest.mark.parametrize("N", [1, 2, 5, 9, 11, 12, 13])
def test_whole_states_single_and_batched(sre, N, kind):
    import torch
    psi = _state(N, kind)
    t = torch.from_numpy(psi).cuda()
    scaled = [torch.from_numpy(psi * s).cuda() for s in (2.0 ** -90, 1.0, 2.0 ** 60)]
    with sre.Plan(N, "c128", "fp64") as p:
        m = p.m2(t)
        assert abs(m - oracle.m2(psi)) <= 1e-12
        got = p.m2_batched(scaled).tolist()
        assert got == [p.m2(s) for s in scaled]
        # powers of two move the units, not the values: equal but for the log
        assert max(abs(g - m) for g in got) <= 1e-12


@pytest.mark.parametrize("N", [6, 13, 16])
def test_states_without_a_finite_norm(sre, N):
    import torch
    for bad in (float("nan"), float("inf")):
        psi = torch.from_numpy(_state(N, "haar")).cuda()
        psi[3] = bad
        with sre.Plan(N, "c128", "fp64") as p:
            with pytest.raises(sre.SreError) as e:
                p.m2(psi)
            assert e.value.status == 4  # SRE_ENONFINITE
            assert not np.isfinite(p.sum4_range(psi, 0, 4)[0].item())
