"""The element kernel's launch shapes (elements per CTA) on both sides of their
dispatch rules: the shape changes the speed, not the result."""
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


# Chandrashekar form at N = 2: the most elements with 128-thread CTAs, and the next larger mesh
@pytest.mark.parametrize("shape", [(32, 20, 19), (32, 20, 20)])
@pytest.mark.parametrize("physics,surface", [("euler", "lf"), ("ns", "roe")])
def test_chandrashekar_n2_cta_sizes(shape, physics, surface):
    om = O.Mesh(*shape, 2, lo=LO, hi=HI, amp=0.05)
    gm = hs.Mesh(*shape, 2, lo=LO, hi=HI, amp=0.05)
    u0 = random_state(om.shape, seed=3, smooth=True)
    u = torch.from_numpy(u0).cuda()
    r = torch.empty_like(u)
    gm.residual(hs.solver_cfg(physics, surface, "ec", "mixed32", Re=400.0), u, r)
    ref = om.residual(O.Cfg(physics, surface, "ec", Re=400.0), u0)
    assert np.linalg.norm(r.cpu().numpy() - ref) / np.linalg.norm(ref) < TOL
