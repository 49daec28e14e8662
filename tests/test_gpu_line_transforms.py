"""The register-resident line transforms (lengths 16 G, G in 2, 4, 6, 8, 10, 12,
16, and the other products of 2, 3 and 5 from 36 to 240) against the FP64
oracle: every length along an axis of each kind of pass, rows of an odd number
of columns (no column pairs to load at once), more lines than fill the last
block, and fields that are only 4-byte aligned."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
TOL = 1e-5  # the operators' tolerance of the parity tests: FP32 rounding of white noise is ~3e-7


def rel(a, b):
    a = a.cpu().numpy().astype(np.float64)
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.fixture(scope="module")
def claire():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2008_12820_gb300 import claire as C
    return C


def unaligned(a):
    """a CUDA copy of a whose first element lies 4 bytes off a 16-byte boundary"""
    buf = torch.empty(a.size + 1, dtype=torch.float32, device="cuda")
    t = buf[1:].view(a.shape)
    t.copy_(torch.from_numpy(a))
    return t


# (x1, x2, x3): each of the seven lengths on each axis
SHAPES = [(32, 64, 96), (64, 96, 32), (96, 32, 64), (128, 6, 160), (5, 160, 192), (160, 192, 4), (192, 10, 128),
          (4, 128, 256), (256, 5, 15), (6, 256, 27), (160, 9, 25), (32, 96, 45), (128, 64, 9)]
# square planes whose x3 and x2 transforms share a launch
SHAPES += [(5, 32, 32), (32, 64, 64), (9, 96, 96)]
# two-step plans of other lengths: as x1, x2 and x3 each once
OTHER = [36, 40, 45, 48, 50, 54, 60, 72, 75, 80, 90, 100, 108, 120, 135, 144, 150, 180, 200, 216, 225, 240]
SHAPES += [s for n in OTHER for s in ((n, 9, 10), (6, n, 15), (5, 8, n))]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("aligned", [True, False], ids=["aligned", "offset"])
def test_line_transforms(claire, shape, aligned):
    rng = np.random.default_rng(sum(shape))
    f = rng.standard_normal(shape).astype(np.float32)
    v = rng.standard_normal((3,) + shape).astype(np.float32)
    dev = (lambda a: torch.from_numpy(a).cuda()) if aligned else unaligned
    beta, gamma = 1e-2, 1.0
    with claire.Registration(shape, 2, beta, gamma) as reg:
        assert rel(reg.grad(dev(f)), O.grad(f)) < TOL
        assert rel(reg.div(dev(v)), O.div(v)) < TOL
        assert rel(reg.apply_A(dev(v)), O.apply_A(v, beta, gamma)) < TOL
        assert rel(reg.precond(dev(v)), O.apply_Ainv(v, beta, gamma)) < TOL
        out = unaligned(np.zeros_like(v)) if not aligned else torch.empty((3,) + shape, device="cuda")
        reg.precond(dev(v), out=out)
        assert rel(out, O.apply_Ainv(v, beta, gamma)) < TOL
