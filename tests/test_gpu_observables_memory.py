"""Observables and deformation allocate nothing, from the first call on, and
work on lattices too small to lend them a workspace."""
import numpy as np
import pytest

import oracle
from helpers import small_2d
from paper_2604_17463_gb300 import iblb
from paper_2604_17463_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


# The driver hands out small buffers from blocks of 2 MB: so many objects that
# ten kilobytes for each would take another block.
MANY = 300


@pytest.mark.parametrize("call", ["observables", "deformation"])
def test_simulation_calls_allocate_nothing(call):
    wl = small_2d()
    sims = [iblb.Simulation.from_workload(wl) for _ in range(MANY)]
    getattr(sims[0], call)()  # kernels are loaded with their first launch
    before = free_bytes()
    for s in sims[1:]:
        getattr(s, call)()
    assert free_bytes() == before
    for s in sims:
        s.close()


def test_batch_observables_allocate_nothing():
    wl = small_2d()
    batches = [iblb.Batch(wl.lattice, iblb.FP64, 1 << 21, max_slots=1) for _ in range(MANY)]
    slots = [b.admit_workload(wl, n_steps=4) for b in batches]
    batches[0].observables(slots[0])
    before = free_bytes()
    for b, k in zip(batches[1:], slots[1:]):
        b.observables(k)
    assert free_bytes() == before
    for b in batches:
        b.close()


@pytest.mark.parametrize("nx,ny", [(14, 13), (14, 15), (32, 30), (32, 31)])
def test_small_lattices(nx, ny):
    # 13 to 31 band segments: no block, one, or two of the workspace fit in
    # their list; 600 nodes ask for three
    nodes = W.circle(600, 4.0, (nx / 2.0 + 0.2, W.WALL_PLANE + 5.2))
    kw = dict(tau=0.9, sigma=1e-3, xi=1.0, theta_eq_deg=60.0)
    g = iblb.Simulation(iblb.D2Q9, nx, ny, **kw)
    o = oracle.Sim(oracle.D2Q9, nx, ny, **kw)
    g.set_interface(nodes)
    o.set_interface(nodes)
    a, b = g.observables(), o.observables()
    for k in ("mass", "volume", "height", "d_min", "radius"):
        assert np.isclose(a[k], b[k], rtol=1e-11, atol=1e-11), k
    assert np.allclose(a["centre"], b["centre"], rtol=1e-11, atol=1e-11)
    d = g.deformation()
    # a polygon of 600 sides: its area and semi-axes are the circle's to 2e-5
    assert np.isclose(d["volume"], np.pi * 16.0, rtol=1e-4) and d["D"] < 1e-9
    assert np.isclose(d["r1"], 4.0, rtol=1e-4) and np.isclose(d["r3"], 4.0, rtol=1e-4)
    g.step(3)
    g.observables()
    g.step(2)
    g.sync()
    g.close()
    o.close()
