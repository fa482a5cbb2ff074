"""The lengths of a ring's segments (chi of the nodal forces) are correctly
rounded roots in every storage form, whichever arithmetic they come from."""
import numpy as np
import pytest

from paper_2604_17463_gb300 import iblb
from paper_2604_17463_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gs", [0.0, 1e-3])
@pytest.mark.parametrize("N", [20, 213, 2000])
@pytest.mark.parametrize("storage", [iblb.FP64, iblb.FP32_DEV])
def test_lengths_are_correctly_rounded(storage, N, gs):
    # binary16 storage takes a root and a division, both correctly rounded
    rng = np.random.default_rng(N)
    nodes = W.circle(N, 80.0, (128.2, 90.1)) + rng.uniform(-1e-2, 1e-2, (N, 2))
    got = []
    for st in (storage, iblb.FP16_DEV):
        s = iblb.Simulation(iblb.D2Q9, 256, 192, tau=0.9, sigma=1e-3, xi=1.0, theta_eq_deg=60.0,
                            shear_modulus=gs, storage=st)
        s.set_interface(nodes)
        got.append(s.nodal_forces())
        s.close()
    assert np.array_equal(got[0][2], got[1][2])
    # forces and normals: a few roundings of the unit tangents apart
    assert np.max(np.abs(got[0][0] - got[1][0])) <= 8 * 2.0 ** -52 * 1e-3
    assert np.max(np.abs(got[0][1] - got[1][1])) <= 8 * 2.0 ** -52


@pytest.mark.parametrize("storage", [iblb.FP64, iblb.FP32_DEV, iblb.FP16_DEV])
def test_length_of_a_degenerate_segment(storage):
    # two nodes in one place (their tangent has no direction, their distance is
    # zero) and two a distance apart whose square is a subnormal number
    nodes = W.circle(12, 8.0, (20.0, 15.0))
    nodes[4] = nodes[3]
    nodes[8] = (0.0, 12.0)
    nodes[9] = (1e-160, 12.0)
    s = iblb.Simulation(iblb.D2Q9, 40, 30, tau=0.9, sigma=1e-3, wetting=False, storage=storage)
    s.set_interface(nodes)
    chi = s.nodal_forces()[2]
    s.close()
    d = np.linalg.norm(np.roll(nodes, -1, 0) - nodes, axis=1)
    assert np.all(np.isfinite(chi))
    assert np.allclose(chi, d + np.roll(d, 1), rtol=1e-15, atol=0)
