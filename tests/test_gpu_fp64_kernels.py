"""FP64 kernels at the edges of their arithmetic: every branch of the
logarithmic mean, and the range test of the reciprocal and square-root steps."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

hs = pytest.importorskip("paper_2206_09733_gb300")

LO, HI = (0.0, 0.0, 0.0), (10.0, 10.0, 10.0)
TOL = 1e-12   # relative to the oracle, as for every well-conditioned FP64 residual


def gpu_residual(gm, gc, u0):
    import torch
    u = torch.from_numpy(u0).cuda()
    r = torch.empty_like(u)
    gm.residual(gc, u, r)
    torch.cuda.synchronize()
    return r.cpu().numpy()


def two_level_state(shape, ratio, seed):
    """rho and p take one of two values `ratio` apart at each node (and a
    velocity of O(1)), so every two-point mean sees equal values or that ratio."""
    rng = np.random.default_rng(seed)
    dims = (shape[0],) + tuple(shape[2:])
    rho = np.where(rng.random(dims) < 0.5, 1.0, ratio)
    p = np.where(rng.random(dims) < 0.5, 1.0, ratio)
    v = rng.uniform(-0.5, 0.5, size=(3,) + dims)
    u = np.empty(shape)
    u[:, 0] = rho
    for c in range(3):
        u[:, 1 + c] = rho * v[c]
    u[:, 4] = p / 0.4 + 0.5 * rho * (v ** 2).sum(0)
    return u


def ratio_of(u):
    """a/b with ((a-b)/(a+b))^2 = u."""
    f = np.sqrt(u)
    return (1 + f) / (1 - f)


@pytest.mark.parametrize("u", [1e-12, 0.99e-4, 1.01e-4, 0.0399, 0.0401, 0.5])
@pytest.mark.parametrize("N,surface,volume", [(3, "lf", "ec"), (4, "ec", "ec"), (2, "matrix", "ir")])
def test_logarithmic_mean_branches(N, surface, volume, u):
    om = O.Mesh(2, 2, 3, N, lo=LO, hi=HI, amp=0.05)
    gm = hs.Mesh(2, 2, 3, N, lo=LO, hi=HI, amp=0.05)
    u0 = two_level_state(om.shape, ratio_of(u), seed=N)
    ref = om.residual(O.Cfg("euler", surface, volume), u0)
    out = gpu_residual(gm, hs.solver_cfg("euler", surface, volume, "fp64"), u0)
    assert np.linalg.norm(out - ref) / np.linalg.norm(ref) < TOL


@pytest.mark.parametrize("shift", [-1000, 0, 1000])
@pytest.mark.parametrize("surface,volume", [("lf", "standard"), ("roe", "ec"), ("rusanov", "kg"), ("ldroe", "pirozzoli")])
def test_states_near_the_ends_of_the_exponent_range(surface, volume, shift):
    """The Euler fluxes are linear in a common factor of (rho, rho v, rho e); a
    power of two is an exact one."""
    om = O.Mesh(2, 3, 2, 3, lo=LO, hi=HI, amp=0.05)
    gm = hs.Mesh(2, 3, 2, 3, lo=LO, hi=HI, amp=0.05)
    u0 = two_level_state(om.shape, 1.3, seed=9)
    ref = om.residual(O.Cfg("euler", surface, volume), u0)
    out = gpu_residual(gm, hs.solver_cfg("euler", surface, volume, "fp64"), np.ldexp(u0, shift))
    assert np.linalg.norm(np.ldexp(out, -shift) - ref) / np.linalg.norm(ref) < TOL
