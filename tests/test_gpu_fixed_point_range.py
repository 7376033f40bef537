"""The FP64 mode at norms where a power of the fixed-point unit leaves the range
of a double although the sum of powers does not.  Scaling a state by a power of
two is exact in every step, so its entropy moves by the rounding of the three
logarithms alone (each below 2^11 in size: 3 * 2^-42, over alpha - 1)."""
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


@pytest.mark.parametrize("N", [6, 13, 14, 15])
@pytest.mark.parametrize("alpha,log2_scale", [(2, 126.5), (2, -126.5), (5, 50), (16, 15.5), (16, -15.5)])
def test_entropy_of_scaled_states(sre, N, alpha, log2_scale):
    import torch
    v = W.product_state(N, 3 + N)[0]
    if log2_scale % 1:  # the half power goes into both states
        v, log2_scale = v * 2.0 ** 0.5, log2_scale - 0.5
    psi = torch.from_numpy(v).cuda()
    with sre.Plan(N, "c128", "fp64") as p:
        want = p.m_alpha(psi, alpha)
        got = p.m_alpha(psi * 2.0 ** log2_scale, alpha)
    assert abs(got - want) <= 2.0 ** -40, (got, want)
