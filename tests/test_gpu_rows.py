"""The N = 7 kernels with four nodes per thread (mixed path: BR1 gradients of
every form, element kernel of the standard form) on the smallest and uneven
meshes, where an element is its own neighbour, and as a Runge-Kutta step."""
import numpy as np
import pytest

import oracle as O
from tests.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2206_09733_gb300 as hs  # noqa: E402

LO, HI = (-np.pi,) * 3, (np.pi,) * 3
# FP32 flux arithmetic on smooth states of O(1): the bar of the mixed path's other parity tests
TOL = 1e-5


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 1, 3)])
@pytest.mark.parametrize("physics,surface,volume", [("euler", "lf", "standard"), ("ns", "roe", "standard"),
                                                    ("ns", "roe", "ec")])
def test_n7_residual_and_step(shape, physics, surface, volume):
    om = O.Mesh(*shape, 7, lo=LO, hi=HI, amp=0.05)
    gm = hs.Mesh(*shape, 7, lo=LO, hi=HI, amp=0.05)
    u0 = random_state(om.shape, seed=5, smooth=True)
    oc = O.Cfg(physics, surface, volume, Re=400.0)
    gc = hs.solver_cfg(physics, surface, volume, "mixed32", Re=400.0)
    u = torch.from_numpy(u0).cuda()
    r = torch.empty_like(u)
    gm.residual(gc, u, r)
    ref = om.residual(oc, u0)
    torch.cuda.synchronize()
    assert np.linalg.norm(r.cpu().numpy() - ref) / np.linalg.norm(ref) < TOL
    g = torch.zeros_like(u)
    gm.rk3_step(gc, u, g)
    uo, go = u0.copy(), np.zeros_like(u0)
    om.rk3_step(oc, uo, go)
    torch.cuda.synchronize()
    # the increment carries the residual's error, the state accumulates in FP64
    assert np.linalg.norm((u.cpu().numpy() - u0) - (uo - u0)) / np.linalg.norm(uo - u0) < TOL
