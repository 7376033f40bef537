"""The one-kernel call of an FP32 state with N <= 12: the norm, the sums and the
result come from the transform's own CTAs.  Sizes below, at and above one norm
block of 256 entries, one tile and many; repeated calls; bad entries at the
ends of a state.  The batch path forms the same partials in separate kernels:
equal bit for bit."""
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


@pytest.mark.parametrize("N", [1, 2, 6, 7, 8, 9, 11, 12])
def test_small_call(sre, N):
    import torch
    psi = torch.from_numpy(3 * W.haar_state(N, 80 + N, np.complex64)).cuda()
    d = 1 << N
    with sre.Plan(12, "c64") as p:
        want = p.m2_batched([psi, psi]).tolist()
        assert [p.m2(psi), p.m2(psi)] == want
        assert p.m2_host(psi.cpu().pin_memory()) == want[0]
        a, b = p.sum4_range(psi, 0, d // 2).tolist(), p.sum4_range(psi, d // 2, d).tolist()
        assert a[1] == b[1]
        for t in (0, d - 1):
            bad = psi.clone()
            bad[t] = complex(float("inf"), 0) if t else complex(0, float("nan"))
            with pytest.raises(sre.SreError) as e:
                p.m2(bad)
            assert e.value.status == 4  # SRE_ENONFINITE
        with pytest.raises(sre.SreError) as e:
            p.m2(torch.zeros_like(psi))
        assert e.value.status == 3  # SRE_EZERO
        assert p.m2(psi) == want[0]
