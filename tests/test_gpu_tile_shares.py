"""Semi-Lagrangian steps on grids whose tiles (32 x 8 x 4 voxels) do not divide
evenly among the resident blocks, with two, three and four tiles a block and one
more in some: every tile is stepped once."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2008_12820_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = 1e-5  # one FP32 operator application, as in the parity tests


# tiles: 960, 1400; resident blocks of the steps: 456 and (with a body force) 304
@pytest.mark.parametrize("shape", [(45, 75, 250), (100, 108, 128)], ids=lambda s: "x".join(map(str, s)))
def test_state_and_matvec(shape):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2008_12820_gb300 import claire as C
    # beta A is negligible: the steps alone are compared
    nt, beta, gamma = 3, 1e-8, 0.0
    d = synth.sinusoid_pair(shape, 1000)
    v = (0.7 * d["v_true"]).astype(np.float32)
    vt = synth.smooth_direction(shape, 11)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    rel = lambda a, b: np.linalg.norm(a.cpu().numpy().astype(np.float64) - b) / np.linalg.norm(b)
    P = O.Problem(d["m0"], d["m1"], nt, beta, gamma)
    _, _, _, m_ref = P.objective(v, want_m_final=True)
    P.linearize(v)
    with C.Registration(shape, nt, beta, gamma) as reg:
        reg.set_images(dev(d["m0"]), dev(d["m1"]))
        assert rel(reg.forward(dev(v))[0], m_ref) < TOL
        reg.linearize(dev(v))
        assert rel(reg.hess_matvec(None, dev(vt)), P.matvec(vt)) < TOL
