"""The finite-difference derivatives on grids large enough for blocks that walk
several planes along x1 (16, 8 or 4, the last block fewer), against the FP64
oracle, FP32 and FP16 output."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
TOL = 1e-6          # FP32: nine roundings of at most 1.2e-7 half the time each way, about 5e-7 of white noise
TOL16 = 2.0 ** -11  # and the rounding of a stored FP16 value

# x1 planes a block: 16 (75 = 4 * 16 + 11), 8 (150 = 18 * 8 + 6), 4 (150 = 37 * 4 + 2)
SHAPES = [(75, 250, 250), (150, 100, 162), (150, 100, 108)]


def rel(a, b):
    a = a.cpu().numpy().astype(np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_fd8_march(shape):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2008_12820_gb300 import claire as C
    rng = np.random.default_rng(3)
    v = rng.standard_normal((3,) + shape).astype(np.float32)
    dv = torch.from_numpy(v).cuda()
    grad = O.grad_fd8(v[0])
    with C.Registration(shape, 1, 1e-2, 1.0) as reg:
        reg.set_discretization("linear", "fd8")
        assert rel(reg.grad(dv[0]), grad) < TOL
        assert rel(reg.div(dv), O.div_fd8(v)) < TOL
    # the FP16 form stores grad m^0 of the template
    with C.Registration(shape, 1, 1e-2, 1.0, precision="fp16") as reg:
        reg.set_discretization("linear", "fd8")
        reg.set_images(dv[0].contiguous(), dv[1].contiguous())
        reg.linearize(torch.zeros_like(dv))
        assert rel(reg.field("gradm", 0), grad) < TOL + TOL16
