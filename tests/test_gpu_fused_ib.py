"""Fused IB kernels and the default launch shape: a chunk of graph-replayed
steps (one ring kernel per step, node forces and spread of a mesh in one
kernel) against the separate kernels of the profiled steps, at ring sizes
around the 30 nodes a warp owns and at odd and even step counts (the ring's
positions change buffers with every step but a chunk's first); and the default
shape of 2D binary16 against the pipelined kernel."""
import numpy as np
import pytest

from helpers import small_2d, small_3d
from paper_2604_17463_gb300 import iblb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,tol", [(iblb.FP64, 1e-13), (iblb.FP32_DEV, 2e-6)])
@pytest.mark.parametrize("N,chunks", [(29, (16,)), (30, (17, 3)), (31, (33, 16)), (60, (31,)), (61, (64, 2)), (150, (19, 32))])
def test_ring_chunks_match_separate_kernels(storage, tol, N, chunks):
    wl = small_2d(nx=64, ny=40, N=N)
    a = iblb.Simulation.from_workload(wl, storage=storage)
    b = iblb.Simulation.from_workload(wl, storage=storage)
    for n in chunks:
        a.step(n)
        b.step_profiled(n)
    ra, ua, qa = a.fields()
    rb, ub, qb = b.fields()
    # node displacements are < 1 lu and every term is the same arithmetic: the
    # two differ by the order of the additions in the spread
    assert np.max(np.abs(ua - ub)) <= tol * max(np.max(np.abs(ub)), 1e-3)
    assert np.max(np.abs(qa - qb)) <= tol
    a.close()
    b.close()


@pytest.mark.parametrize("storage,tol", [(iblb.FP64, 1e-13), (iblb.FP32_DEV, 2e-6)])
def test_mesh_chunks_match_separate_kernels(storage, tol):
    wl = small_3d(n=30, nz=22, R=7.0, level=3)
    a = iblb.Simulation.from_workload(wl, storage=storage)
    b = iblb.Simulation.from_workload(wl, storage=storage)
    a.step(35)
    b.step_profiled(35)
    _, ua, qa = a.fields()
    _, ub, qb = b.fields()
    assert np.max(np.abs(ua - ub)) <= tol * np.max(np.abs(ub))
    assert np.max(np.abs(qa - qb)) <= tol
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny", [(64, 40), (96, 33), (512, 60)])
def test_default_binary16_ring_has_the_pipelined_bits(nx, ny):
    wl = small_2d(nx=nx, ny=ny)
    out = []
    for pipelined in (False, True):
        g = iblb.Simulation.from_workload(wl, storage=iblb.FP16_DEV, deterministic_spread=True)
        if pipelined:
            g.set_tuning(1)
            assert g.variant == 1
        g.step(25)
        out.append(g.populations())
        g.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("which", ["2d", "3d"])
@pytest.mark.parametrize("storage,tol", [(iblb.FP64, 1e-12), (iblb.FP32_DEV, 1e-5)])
def test_batch_in_two_parts_matches_single_engine(which, storage, tol):
    # enough cells for two parts; the slots end at different steps, so the
    # parts are cut anew, down to one slot in one part
    if which == "2d":
        wls = [small_2d(nx=nx, ny=ny, R=9.0, N=N) for nx, ny, N in ((700, 300, 61), (33, 40, 29), (260, 330, 90))]
    else:
        wls = [small_3d(n=n, nz=nz, R=7.0, level=2) for n, nz in ((80, 40), (24, 22), (40, 40))]
    steps = (40, 17, 33)
    b = iblb.Batch(wls[0].lattice, storage, 1 << 30, max_slots=4)
    slots = [b.admit_workload(w, n_steps=n) for w, n in zip(wls, steps)]
    b.run(64)
    for w, n, s in zip(wls, steps, slots):
        _, u, q = b.fields(s)
        g = iblb.Simulation.from_workload(w, storage=storage)
        g.step(n)
        _, ug, qg = g.fields()
        g.close()
        assert np.linalg.norm(u - ug) <= tol * np.linalg.norm(ug)
        assert np.max(np.abs(q - qg)) <= tol * 10
    b.close()


@pytest.mark.parametrize("which", ["2d", "3d"])
def test_observables_over_many_blocks(which):
    # more nodes than one block takes in a pass, against the oracle's estimator
    import oracle
    from paper_2604_17463_gb300 import workloads as W
    if which == "2d":
        wl = W.spreading_2d_2048x512(downscale=4)
        nodes = W.truncated_circle(2000, 50.0, 150.0, W.WALL_PLANE + wl.xi, 256.0)
        faces = None
    else:
        wl = small_3d(n=64, nz=48, R=15.0, level=2)
        nodes, faces = W.icosphere(5, 15.0, (32.3, 31.8, W.WALL_PLANE + 17.0))
    kw = dict(tau=wl.tau, sigma=wl.sigma, xi=wl.xi, theta_eq_deg=wl.theta_eq_deg)
    g = iblb.Simulation(wl.lattice, wl.nx, wl.ny, wl.nz, **kw)
    o = oracle.Sim(wl.lattice, wl.nx, wl.ny, wl.nz, **kw)
    g.set_interface(nodes, faces)
    o.set_interface(nodes, faces)
    a, b = g.observables(), o.observables()
    # at rest every density is 1: the mass is the number of fluid cells, exactly
    assert a["mass"] == wl.fluid_cells
    for k in ("volume", "height", "d_min", "radius"):
        assert np.isclose(a[k], b[k], rtol=1e-11, atol=1e-11, equal_nan=True), k
    # the whole sphere meets the plane of its lowest node at 180 degrees, where
    # the angle and the contact radius are the square roots of rounding errors:
    # their cosine and square are compared, and the film (the mean over the
    # nodes within half that radius) where there is a contact radius
    if b["r_cl"] > 1e-3:
        assert np.isclose(a["film"], b["film"], rtol=1e-11, atol=1e-11, equal_nan=True)
    assert np.isclose(np.cos(np.radians(a["theta_deg"])), np.cos(np.radians(b["theta_deg"])), rtol=0, atol=1e-11)
    assert np.isclose(a["r_cl"] ** 2, b["r_cl"] ** 2, rtol=0, atol=1e-11 * b["radius"] ** 2)
    assert np.allclose(a["centre"], b["centre"], rtol=1e-11, atol=1e-11)
    g.close()
    o.close()


@pytest.mark.parametrize("heap", [31, 33, 200, 300])
def test_ordered_spread_sorts_crowded_bins(heap):
    # `heap` nodes of a ring within one bin of the ordered spread: the force
    # field is that of the atomic spread up to the order of the additions, and
    # the same twice
    import math
    n = heap + 60
    a = np.concatenate([np.linspace(-0.02, 0.02, heap, endpoint=False),
                        np.linspace(0.02, 2 * math.pi - 0.02, 60, endpoint=False)])
    nodes = np.stack([32.4 + 12 * np.cos(a), 16.3 + 12 * np.sin(a)], axis=1)
    out = []
    for ordered in (True, True, False):
        g = iblb.Simulation(iblb.D2Q9, 64, 40, wetting=False, sigma=1e-3, deterministic_spread=ordered)
        g.set_interface(nodes)
        out.append(g.force_field())
        g.close()
    assert np.array_equal(out[0], out[1])
    assert np.max(np.abs(out[0] - out[2])) <= 1e-12 * np.max(np.abs(out[2]))
