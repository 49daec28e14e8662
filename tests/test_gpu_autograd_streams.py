"""Differentiable transport without host synchronizations: the device mismatch
equals the host one, and a context on a stream of its own gives the same values
as one on the caller's stream."""
import pytest
import torch

from paper_2008_12820_gb300 import synth

pytestmark = pytest.mark.gpu
SHAPE, NT = (32, 40, 48), 4


@pytest.fixture(scope="module")
def problem():
    import __graft_entry__
    __graft_entry__.build()
    d = synth.sinusoid_pair(SHAPE, 1000)
    return {k: torch.from_numpy(d[k]).cuda() for k in ("m0", "m1", "v_true")}


def step(C, p, stream, stride, weight):
    from paper_2008_12820_gb300.autograd import transport_mismatch
    with C.Registration(SHAPE, NT, 1e-2, 1.0, stream=stream) as reg:
        reg.set_images(p["m0"], p["m1"])
        v = (0.7 * p["v_true"]).requires_grad_(True)
        torch.cuda.synchronize()
        mis, m = transport_mismatch(v, reg, stride)
        loss = mis + weight * m.square().sum()
        loss.backward()
        out = mis.detach().clone(), m.detach().clone(), v.grad.clone()
        torch.cuda.synchronize()
        host_m, host_mis = reg.mismatch_forward(v.detach(), stride)
        assert mis.dtype == torch.float64 and float(mis.detach()) == host_mis
        assert torch.equal(host_m, out[1])
        return out


@pytest.mark.parametrize("stride", [1, 2, 3, 4])
@pytest.mark.parametrize("weight", [0.0, 0.1])
def test_own_stream_equals_current_stream(problem, stride, weight):
    from paper_2008_12820_gb300 import claire as C
    a = step(C, problem, None, stride, weight)
    b = step(C, problem, torch.cuda.Stream(), stride, weight)
    for x, y in zip(a, b):
        assert torch.equal(x, y)


def test_device_mismatch_needs_a_forward(problem):
    from paper_2008_12820_gb300 import claire as C
    with C.Registration(SHAPE, NT, 1e-2, 1.0) as reg:
        out = torch.empty((), dtype=torch.float64, device="cuda")
        with pytest.raises(C.ClaireError) as e:
            reg._c("claire_mismatch_device", out.data_ptr())
        assert e.value.code == 4
