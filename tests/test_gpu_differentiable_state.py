"""State that the differentiable transport keeps between calls: reductions that
a call leaves in flight on its stream."""
import pytest
import torch

from paper_2008_12820_gb300 import synth

pytestmark = pytest.mark.gpu
SHAPE, NT = (32, 40, 48), 4
DELAY = 100_000_000  # GPU cycles (about 50 ms), far longer than the calls under test


@pytest.fixture(scope="module")
def C():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2008_12820_gb300 import claire
    return claire


@pytest.fixture(scope="module")
def problem():
    d = synth.sinusoid_pair(SHAPE, 1000)
    return {k: torch.from_numpy(d[k]).cuda() for k in ("m0", "m1", "v_true")}


def test_new_stream_waits_for_a_reduction_in_flight(C, problem):
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    out = torch.zeros((), dtype=torch.float64, device="cuda")
    v = 0.7 * problem["v_true"]
    with C.Registration(SHAPE, NT, 1e-2, 1.0, stream=a) as reg:
        torch.cuda.synchronize()
        reg.set_images(problem["m0"], problem["m1"])
        _, mis = reg.mismatch_forward(v)
        with torch.cuda.stream(a):
            torch.cuda._sleep(DELAY)
            delayed = a.record_event()
        reg._c("claire_mismatch_device", out.data_ptr())
        assert not delayed.query()
        reg._c("claire_set_stream", b.cuda_stream)
        b.synchronize()
        assert delayed.query()
        # and the context reduces as before on its new stream
        torch.cuda.synchronize()
        assert float(out) == mis and reg.mismatch_forward(v)[1] == mis
