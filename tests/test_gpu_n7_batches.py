"""N = 7, mixed path: launches over few elements take other kernels than larger
ones (two elements per SM is the line), and a solve may run alone or in a
batch: the results are the same either way, and match the oracle on both
sides of the line."""
import time

import numpy as np
import pytest

import oracle as O
from tests.inputs import random_state

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2206_09733_gb300 as hs  # noqa: E402

LO, HI = (-np.pi,) * 3, (np.pi,) * 3
FORMS = [("euler", "lf", "standard"), ("ns", "roe", "standard"), ("ns", "roe", "ec")]
# FP32 flux arithmetic on smooth states of O(1): the bar of the mixed path's other parity tests
TOL = 1e-5


def serve(shapes, cfg, amp, steps, mode="grid"):
    """Final states of Taylor-Green solves on the given boxes, submitted together."""
    srv = hs.Server(launch_mode=mode)
    outs, tickets = [], []
    for shape in shapes:
        outs.append(np.zeros((int(np.prod(shape)), 5, 8, 8, 8)))
        tickets.append(srv.submit(hs.mesh_desc(*shape, 7, lo=LO, hi=HI, amp=amp), cfg, hs.ic_desc("tgv", 1.4, 0.1),
                                  n_steps=steps, result=outs[-1]))
    t0 = time.time()
    for t in tickets:
        while True:
            st, _ = srv.poll(t)
            if st != hs.PENDING:
                break
            assert time.time() - t0 < 120
            time.sleep(0.002)
        assert st == hs.OK
    srv.close()
    return outs


@pytest.mark.parametrize("physics,surface,volume", FORMS)
def test_alone_equals_batched(physics, surface, volume):
    # alone: 24, 125 (few elements), 336 (more than two per SM); together 485
    shapes = [(3, 2, 4), (6, 7, 8), (5, 5, 5)]
    cfg = hs.solver_cfg(physics, surface, volume, "mixed32", Re=400.0, Ma=0.1, cfl=0.5)
    outs = serve(shapes, cfg, 0.05, 4)
    for shape, out in zip(shapes, outs):
        m = hs.Mesh(*shape, 7, lo=LO, hi=HI, amp=0.05)
        u = m.init_state(m.empty_state(), "tgv", 1.4, 0.1)
        m.rk3_run(cfg, u, torch.zeros_like(u), 4)
        assert np.array_equal(u.cpu().numpy(), out), shape


# one element more than the few-element kernels take, and the most they take
@pytest.mark.parametrize("shape", [(5, 61, 1), (8, 19, 2)])
@pytest.mark.parametrize("physics,surface,volume", FORMS)
def test_both_sides_of_the_line_match_the_oracle(shape, physics, surface, volume):
    om = O.Mesh(*shape, 7, lo=LO, hi=HI, amp=0.05)
    gm = hs.Mesh(*shape, 7, lo=LO, hi=HI, amp=0.05)
    u0 = random_state(om.shape, seed=5, smooth=True)
    oc = O.Cfg(physics, surface, volume, Re=400.0)
    gc = hs.solver_cfg(physics, surface, volume, "mixed32", Re=400.0)
    u = torch.from_numpy(u0).cuda()
    r = torch.empty_like(u)
    gm.residual(gc, u, r)
    ref = om.residual(oc, u0)
    assert np.linalg.norm(r.cpu().numpy() - ref) / np.linalg.norm(ref) < TOL
    gm.rk3_step(gc, u, torch.zeros_like(u))
    uo = u0.copy()
    om.rk3_step(oc, uo, np.zeros_like(uo))
    assert np.linalg.norm((u.cpu().numpy() - u0) - (uo - u0)) / np.linalg.norm(uo - u0) < TOL


@pytest.mark.parametrize("physics,surface,volume", FORMS)
def test_persistent_grids_equal_cta_grids(physics, surface, volume):
    """More elements (1,190) than CTAs fit on the GPU at once, in a batch of three:
    the persistent CTAs walk several tiles.  The kernels are instantiations of
    their own, in which the compiler may fuse the FP32 multiply-adds differently:
    equal to the FP32 rounding of the residual, as for the other degrees."""
    shapes = [(9, 9, 9), (5, 5, 5), (6, 7, 8)]
    cfg = hs.solver_cfg(physics, surface, volume, "mixed32", Re=400.0, Ma=0.1, cfl=0.5)
    for a, b in zip(serve(shapes, cfg, 0.05, 3), serve(shapes, cfg, 0.05, 3, "persistent")):
        assert np.abs(a - b).max() <= 1e-7 * np.abs(a).max()
