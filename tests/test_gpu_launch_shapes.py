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


def cached(path):
    import json
    return json.loads(path.read_text())


def test_tuning_reports_and_keeps_shapes_that_run(tmp_path, monkeypatch):
    """The Chandrashekar kernel at N = 3 and 4 takes at most 128 threads, and a
    choice for it is none for the other split forms."""
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("HS3D_TUNE_CACHE", str(cache))
    ns = dict(precision="mixed32", Re=400.0)
    for N, E, most in ((3, 9, 2), (4, 7, 1)):
        m = hs.Mesh(E, E, E, N, lo=LO, hi=HI, amp=0.05)
        grad, elem = m.autotune(hs.solver_cfg("ns", "roe", "ec", **ns))
        assert 1 <= elem <= most and grad * (N + 1) ** 3 <= 256
        assert cached(cache)[f"N{N}_p1_k1"] == elem and cached(cache)[f"N{N}_p1_k0"] == grad
    m = hs.Mesh(9, 9, 9, 3, lo=LO, hi=HI, amp=0.05)
    before = cached(cache)
    _, elem = m.autotune(hs.solver_cfg("ns", "roe", "kg", **ns))
    after = cached(cache)
    assert after["N3_p1_k2"] == elem and after["N3_p1_k1"] == before["N3_p1_k1"]


@pytest.mark.parametrize("precision,volume,nodes", [("mixed32", "ec", "lobatto"), ("fp64", "kg", "lobatto"),
                                                    ("mixed32", "standard", "gauss")])
def test_tuning_on_a_mesh_too_small_for_the_shapes_to_differ(precision, volume, nodes, tmp_path, monkeypatch):
    """Such a mesh's launches stay spread (one element per CTA), the choice kept for
    larger ones is within the largest CTA, and results stay the same bit for bit."""
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("HS3D_TUNE_CACHE", str(cache))
    m = hs.Mesh(3, 3, 3, 2, lo=LO, hi=HI, amp=0.05, nodes=nodes)
    cfg = hs.solver_cfg("ns", "roe", volume, precision, Re=400.0)
    u = torch.from_numpy(random_state(m.shape, seed=4, smooth=True)).cuda()
    r0, r1 = torch.empty_like(u), torch.empty_like(u)
    m.residual(cfg, u, r0)
    assert m.autotune(cfg) == (1, 1)
    kept = cached(cache)
    assert all(1 <= v and (2 < int(k[1]) or v * 27 <= 256) for k, v in kept.items() if k.startswith("N2"))
    m.residual(cfg, u, r1)
    assert torch.equal(r0, r1)


# buckets of about 144 elements, three to a CTA (576 elements share the SMs), and of a few
@pytest.mark.parametrize("shape", [(8, 8, 9), (3, 2, 2)])
@pytest.mark.parametrize("precision,volume", [("mixed32", "ec"), ("mixed32", "standard"), ("fp64", "ec")])
def test_degree_buckets_side_by_side(shape, precision, volume):
    # (mixed: the bar of the mixed path's other mortar tests)
    from tests import inputs as I
    from tests.test_gpu_pmesh import TOLMIX, pair, rel, to_dev, to_host
    deg = I.random_degrees(int(np.prod(shape)), seed=11, lo=2, hi=5)
    om, gm = pair(*shape, deg, amp=0.05)
    u0 = I.random_state_blocks(deg, seed=43, smooth=True)
    ref = om.residual(O.Cfg("ns", "roe", volume, Re=400.0), u0)
    ud = to_dev(om, gm, u0)
    r = torch.zeros_like(ud)
    gm.residual(hs.solver_cfg("ns", "roe", volume, precision, Re=400.0), ud, r)
    assert rel(to_host(om, gm, r), ref) <= (TOLMIX if precision == "mixed32" else 1e-12)
