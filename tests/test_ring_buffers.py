"""The fused ring kernel moves the nodes into the nodal forces' array, so that a
2D interface takes two arrays of its nodes in every storage form, and the calls
that read positions or forces between steps find them."""
import numpy as np
import pytest

from helpers import small_2d
from paper_2604_17463_gb300 import iblb


@pytest.mark.parametrize("storage", [iblb.FP64, iblb.FP32_DEV, iblb.FP16_DEV])
def test_slot_takes_positions_and_forces(storage):
    cfg = iblb.make_config(iblb.D2Q9, 96, 48, storage=storage)
    # both arrays are multiples of the arena's 256 bytes
    per_node = (iblb.Batch.footprint(cfg, 2048) - iblb.Batch.footprint(cfg, 1024)) / 1024
    assert per_node == 2 * 16


@pytest.mark.gpu
@pytest.mark.parametrize("storage,tol", [(iblb.FP64, 1e-12), (iblb.FP32_DEV, 2e-6)])
def test_reads_between_fused_steps(storage, tol):
    wl = small_2d(nx=64, ny=40, N=67)
    a = iblb.Simulation.from_workload(wl, storage=storage)
    b = iblb.Simulation.from_workload(wl, storage=storage)
    for n in (16, 33, 1, 32, 5, 17):
        a.step(n)
        b.step_profiled(n)
        for x, y in zip(a.nodal_forces(), b.nodal_forces()):
            assert np.max(np.abs(x - y)) <= tol * max(1.0, np.max(np.abs(y)))
        assert np.max(np.abs(a.force_field() - b.force_field())) <= 10 * tol * np.max(np.abs(b.force_field()))
        assert np.max(np.abs(a.fields()[2] - b.fields()[2])) <= tol
    a.close()
    b.close()
