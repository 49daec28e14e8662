"""State that the differentiable transport keeps between calls: reductions that
a call leaves in flight on its stream, and the images of the last forward; and
which of its calls return behind their work."""
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


def test_replaced_images_end_the_mismatch_of_the_last_forward(C, problem):
    """Checkpoints of one pair and the reference image of another belong to no
    mismatch; the upstream gradient of m(1) alone needs neither image."""
    out = torch.zeros((), dtype=torch.float64, device="cuda")
    v = 0.7 * problem["v_true"]
    with C.Registration(SHAPE, NT, 1e-2, 1.0) as reg:
        reg.set_images(problem["m0"], problem["m1"])
        _, mis = reg.mismatch_forward(v)
        of_m1 = reg.mismatch_backward(0.0, problem["m0"])
        both = reg.mismatch_backward(1.0, problem["m0"])
        reg.set_images(problem["m1"], problem["m0"])
        for call in (lambda: reg._c("claire_mismatch_device", out.data_ptr()),
                     lambda: reg.mismatch_backward(1.0), lambda: reg.mismatch_backward(1.0, problem["m0"])):
            with pytest.raises(C.ClaireError) as e:
                call()
            assert e.value.code == 4
        assert torch.equal(reg.mismatch_backward(0.0, problem["m0"]), of_m1)
        reg.set_images(problem["m0"], problem["m1"])
        assert reg.mismatch_forward(v)[1] == mis
        assert torch.equal(reg.mismatch_backward(1.0, problem["m0"]), both)
        reg._c("claire_mismatch_device", out.data_ptr())
        assert float(out) == mis


def test_mismatch_forward_returns_behind_its_work(C, problem):
    """claire_mismatch_forward synchronizes whether or not the mismatch is asked
    for; claire_mismatch_forward_device does not."""
    a = torch.cuda.Stream()
    v = 0.7 * problem["v_true"]
    m, out = torch.empty(SHAPE, device="cuda"), torch.zeros((), dtype=torch.float64, device="cuda")
    with C.Registration(SHAPE, NT, 1e-2, 1.0, stream=a) as reg:
        torch.cuda.synchronize()
        reg.set_images(problem["m0"], problem["m1"])
        ref, mis = reg.mismatch_forward(v)
        args = reg._vec(v), reg._scal(m)
        for name, mismatch, behind in (("claire_mismatch_forward", None, True),
                                       ("claire_mismatch_forward_device", out.data_ptr(), False)):
            m.zero_()
            torch.cuda.synchronize()
            with torch.cuda.stream(a):
                torch.cuda._sleep(DELAY)
            reg._c(name, *args, mismatch, 2)
            assert a.query() is behind
            torch.cuda.synchronize()
            assert torch.equal(m, ref)
        assert float(out) == mis
