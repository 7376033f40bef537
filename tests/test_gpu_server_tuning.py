"""sre_server_set_tuning applies what the caller gives: fields beside the ring
too, with the library's own ring.  Pass-2 items of one tile in place of several
add the split modes' FP32 partial sums in another grouping, which moves the last
places of M2; a server with that tuning gives the plan's value bit for bit."""
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


def test_item_fields_alone_reach_the_units(sre):
    import torch
    N, fields = 17, {"pass2_tiles_log": 0}
    v = W.product_state(N, 500, np.complex64)[0]
    dev = torch.from_numpy(v).cuda()
    with sre.Plan(N, "c64", "fp16_split") as p:
        library = p.m2(dev)
        p.set_tuning(**fields)
        want = p.m2(dev)
    assert want != library, "the state does not tell the two groupings apart"
    with sre.Server(max_inflight=1, max_N=N, mode="fp16_split", slot_scratch_bytes=192 << 20) as srv:
        srv.set_tuning(N, fields)
        assert srv.wait(srv.submit(v), 60000) == want


@pytest.mark.parametrize("mode,N", [("fp16_split", 18), ("fp64", 16), ("fp32", 18)])
def test_library_tuning_of_a_plan_is_taken_and_a_larger_ring_refused(sre, mode, N):
    v = W.haar_state(N, 44, np.complex128 if mode == "fp64" else np.complex64)
    dtype = "c128" if mode == "fp64" else "c64"
    with sre.Plan(N, dtype, mode) as p:
        t = p.get_tuning(N)
    with sre.Server(max_inflight=1, max_N=N, mode=mode, slot_scratch_bytes=96 << 20) as srv:
        srv.set_tuning(N, t)
        srv.wait(srv.submit(v), 120000)
        with pytest.raises(sre.SreError) as e:
            srv.set_tuning(N, {"x_batch_log": 3, "ring_slots": 60, "lag": 20})
        assert e.value.status == 1
