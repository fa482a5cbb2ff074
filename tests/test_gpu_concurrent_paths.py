"""Paths that run beside others: the overlapped step with a viscosity ratio, a
batch of meshes in two parts with one in both parts, and the binary16 bulk
kernel of four cells per thread against the row pairs."""
import numpy as np
import pytest

from helpers import small_3d
from paper_2604_17463_gb300 import iblb

pytestmark = pytest.mark.gpu


def tau_out(tau, lam):
    return 0.5 + (tau - 0.5) / lam


@pytest.mark.parametrize("lam", [0.5, 2.0])
@pytest.mark.parametrize("storage", [iblb.FP64, iblb.FP32_DEV, iblb.FP16_DEV])
def test_overlapped_viscosity_ratio_equals_serial_bitwise(storage, lam):
    # 40 x 40 x 24: FP64 overlaps by default from 2^15 cells; the runs cross
    # the 32-step chunks, and every call starts with a first step
    wl = small_3d(n=40, nz=24, R=7.0)
    out = []
    for overlap in (2, 1, 0):
        g = iblb.Simulation.from_workload(wl, storage=storage, deterministic_spread=True,
                                          tau_out=tau_out(wl.tau, lam))
        g.set_tuning(0, step_overlap=overlap)
        for n in (1, 33, 2):
            g.step(n)
        out.append(g.fields() + (g.populations(),))
        g.close()
    for other in out[1:]:
        for x, y in zip(out[0], other):
            assert np.array_equal(x, y)


@pytest.mark.parametrize("storage,tol", [(iblb.FP64, 1e-12), (iblb.FP32_DEV, 1e-5)])
def test_two_parts_with_viscosity_ratios(storage, tol):
    # 2^18 cells and more in all, so two parts; a ratio on either side of the
    # cut and slots without one, ending at different steps
    sizes = ((64, 40), (24, 22), (64, 40), (40, 24), (24, 22))
    lams = (0.5, None, None, 2.0, 0.5)
    steps = (40, 33, 37, 40, 17)
    wls = [small_3d(n=n, nz=nz, R=7.0, level=2) for n, nz in sizes]
    assert sum(n * n * (nz - 2) for n, nz in sizes) >= 1 << 18
    b = iblb.Batch(wls[0].lattice, storage, 1 << 30, max_slots=8)
    over = [{} if lam is None else {"tau_out": tau_out(w.tau, lam)} for w, lam in zip(wls, lams)]
    slots = [b.admit_workload(w, n_steps=n, **o) for w, n, o in zip(wls, steps, over)]
    b.run(64)
    for w, n, o, s in zip(wls, steps, over, slots):
        _, u, q = b.fields(s)
        g = iblb.Simulation.from_workload(w, storage=storage, **o)
        g.step(n)
        _, ug, qg = g.fields()
        g.close()
        assert np.linalg.norm(u - ug) <= tol * np.linalg.norm(ug)
        assert np.max(np.abs(q - qg)) <= tol * 10
    b.close()


@pytest.mark.parametrize("walls", [True, False])
@pytest.mark.parametrize("nx,ny,nz", [(2, 5, 4), (34, 6, 5), (130, 7, 4), (600, 3, 5), (8, 2, 3)])
@pytest.mark.parametrize("block_x", [64, 128, 256])
def test_four_cells_per_thread_have_the_row_pairs_bits(nx, ny, nz, walls, block_x):
    # a body force that is zero in FP32 keeps the row pairs' kernel, with the
    # values of no force
    f = None
    out = []
    for body in (0.0, 1e-300):
        s = iblb.Simulation(iblb.D3Q19, nx, ny, nz, tau=0.77, walls=walls, wetting=False,
                            storage=iblb.FP16_DEV, body_force=(body, 0.0, 0.0))
        s.set_tuning(3, block_x)
        assert s.variant == 3
        if f is None:
            f = s.populations()
            f = f + np.random.default_rng(nx).uniform(-2e-3, 2e-3, f.shape)
        s.set_populations(f)
        s.step(9)
        out.append((s.populations(),) + s.fields()[:2])
        s.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)
