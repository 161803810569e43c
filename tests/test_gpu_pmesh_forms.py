"""Mixed precision on mortar meshes: every split form with viscosity, whose
element kernel takes the viscous flux of its surface term from its staged
values, and the packed mortar interpolation over degrees 1..7 (odd and even
numbers of nodes), against the oracle."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from tests import inputs as I  # noqa: E402
from tests.test_gpu_pmesh import TOLMIX, cfgs, pair, rel, to_dev, to_host  # noqa: E402


# (curved meshes start at degree 2)
@pytest.mark.parametrize("lo,hi,amp", [(1, 3, 0.0), (2, 7, 0.08)])
@pytest.mark.parametrize("volume", ["ec", "kg", "pirozzoli", "ducros", "morinishi", "ir"])
def test_viscous_split_forms_mixed(volume, lo, hi, amp):
    deg = I.random_degrees(3 * 2 * 3, seed=11, lo=lo, hi=hi)
    om, gm = pair(3, 2, 3, deg, amp=amp)
    oc, gc = cfgs("ns", "roe", volume, "mixed32")
    u = I.random_state_blocks(deg, seed=43, smooth=True)
    ref = om.residual(oc, u)
    ud = to_dev(om, gm, u)
    r = torch.zeros_like(ud)
    gm.residual(gc, ud, r)
    # FP32 flux and mortar arithmetic: the bar of the mixed path's other mortar tests
    assert rel(to_host(om, gm, r), ref) <= TOLMIX
