"""D2Q9 with binary16 storage: the launch shapes that share one arithmetic (the
plain kernel at every block size and the pipelined kernel) give the same bits,
so that reading the launch shape and setting it again changes nothing.  The
ordered spread makes a run a function of its inputs."""
import numpy as np
import pytest

from helpers import small_2d
from paper_2604_17463_gb300 import iblb

pytestmark = pytest.mark.gpu

CASES = {
    "ring": dict(interface=True),
    "ring_body_force": dict(interface=True, body_force=(2e-6, 0.0, 0.0)),
    "free": dict(interface=False),
    "free_body_force": dict(interface=False, body_force=(2e-6, -1e-6, 0.0)),
    "free_periodic": dict(interface=False, walls=False, wetting=False),
}


def run(nx, ny, tuning, interface, steps=40, **over):
    wl = small_2d(nx=nx, ny=ny)
    kw = dict(tau=wl.tau, sigma=wl.sigma, xi=wl.xi, theta_eq_deg=wl.theta_eq_deg)
    kw.update(over)
    s = iblb.Simulation(iblb.D2Q9, nx, ny, storage=iblb.FP16_DEV, deterministic_spread=True, **kw)
    if interface:
        s.set_interface(wl.nodes)
    f = s.populations()
    noise = np.random.default_rng(5).uniform(-2e-3, 2e-3, f.shape)
    s.set_populations(f + noise)
    if tuning == "again":
        t = s.tuning()
        s.set_tuning(**t)
    elif tuning is not None:
        s.set_tuning(**tuning)
        assert s.variant == tuning["variant"]
    s.step(steps)
    out = s.populations()
    s.close()
    return out


@pytest.mark.parametrize("what", list(CASES))
@pytest.mark.parametrize("nx,ny", [(64, 40), (256, 33), (75, 41)])
def test_shapes_of_one_arithmetic_have_the_same_bits(what, nx, ny):
    ref = run(nx, ny, None, **CASES[what])
    shapes = ["again", dict(variant=0, block_x=64), dict(variant=0, block_x=256, streaming_stores=1),
              dict(variant=0, step_overlap=1)]
    if nx % 32 == 0:
        shapes += [dict(variant=1), dict(variant=1, rows_per_tile=1)]
    for t in shapes:
        assert np.array_equal(run(nx, ny, t, **CASES[what]), ref), t
