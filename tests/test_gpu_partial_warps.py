"""Batches whose CTAs end in a partly filled warp (whole elements of 27 or 125
nodes per CTA) and hold elements of two solves: the time step of each solve, and
with it its state, is that of the solve alone."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2206_09733_gb300 as hs  # noqa: E402

LO, HI = (-np.pi,) * 3, (np.pi,) * 3


@pytest.mark.parametrize("N,precision,nodes", [(2, "fp64", "lobatto"), (4, "fp64", "lobatto"), (2, "mixed32", "gauss"),
                                               (4, "mixed32", "gauss"), (2, "fp64", "gauss")])
def test_batched_time_steps(N, precision, nodes):
    # (several elements per CTA from 152 elements per element of a CTA on; odd counts, so
    # that the solves share CTAs)
    shapes = [(9, 9, 9), (7, 5, 3), (2, 2, 2), (11, 9, 7)]
    cfg = hs.solver_cfg("ns", "roe", "standard" if nodes == "gauss" else "ec", precision, Re=400.0, Ma=0.1, cfl=0.5)
    srv = hs.Server()
    outs, tickets = [], []
    for k, shape in enumerate(shapes):
        outs.append(np.zeros((int(np.prod(shape)), 5) + (N + 1,) * 3))
        desc = hs.mesh_desc(*shape, N, lo=LO, hi=HI, amp=0.02 * k, nodes=nodes)
        tickets.append(srv.submit(desc, cfg, hs.ic_desc("tgv", 1.4, 0.1), n_steps=3, result=outs[-1]))
    t0 = time.time()
    for t in tickets:
        while srv.poll(t)[0] == hs.PENDING:
            assert time.time() - t0 < 60
            time.sleep(0.002)
    srv.close()
    for k, (shape, out) in enumerate(zip(shapes, outs)):
        m = hs.Mesh(*shape, N, lo=LO, hi=HI, amp=0.02 * k, nodes=nodes)
        u = m.init_state(m.empty_state(), "tgv", 1.4, 0.1)
        m.rk3_run(cfg, u, torch.zeros_like(u), 3)
        assert np.array_equal(u.cpu().numpy(), out), shape
