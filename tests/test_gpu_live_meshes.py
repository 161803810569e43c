"""Several meshes with per-direction degrees alive at once: creating one must
not change what the kernels of another may use (a function's shared-memory
limit belongs to the function, not to the mesh)."""
import numpy as np
import pytest

from tests import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2206_09733_gb300 as hs  # noqa: E402

LO, HI = (-np.pi,) * 3, (np.pi,) * 3


# highest degree first in every row: 256 thread slots (up to 6 x 6 x 6 nodes), 512 slots (8 x 8 x 8)
@pytest.mark.parametrize("ranges", [((2, 5), (2, 3), (2, 4)), ((2, 7), (6, 6), (2, 4), (2, 2))])
@pytest.mark.parametrize("physics,volume", [("ns", "ec"), ("ns", "ir"), ("euler", "kg"), ("ns", "standard")])
def test_a_later_mesh_leaves_earlier_ones_usable(ranges, physics, volume):
    cfg = hs.solver_cfg(physics, "roe", volume, "fp64", Re=200.0)
    live = []
    for lo, hi in ranges:
        deg = I.random_degree_triples(12, seed=7, lo=lo, hi=hi)
        deg[0] = (hi, hi, hi)
        deg[1] = (hi, lo, hi - 1 if hi > 2 else hi)
        if lo == hi:
            deg[2, 0] = lo - 1      # (equal degrees everywhere would take the bucketed path)
        m = hs.PMesh(3, 2, 2, deg, lo=LO, hi=HI, amp=0.0 if deg.min() < 2 else 0.05)
        u = torch.from_numpy(I.random_state_blocks(deg, seed=3, smooth=True)).cuda()
        r = torch.empty_like(u)
        m.residual(cfg, u, r)
        live.append((m, u, r))
    for m, u, r in live:
        again = torch.empty_like(u)
        m.residual(cfg, u, again)
        assert torch.equal(again, r)
        m.clock(reset=True)
        m.run(cfg, u, torch.zeros_like(u), 2)
        assert m.clock()[1] == 2
