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
