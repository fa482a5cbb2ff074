"""Reading the fields leaves no device memory behind: a program may hold as many
simulations and batches as fit by their own buffers."""
import pytest

from helpers import small_3d
from paper_2604_17463_gb300 import iblb

pytestmark = pytest.mark.gpu


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_simulation_read_keeps_nothing():
    import torch
    torch.cuda.init()
    wl = small_3d(n=128, nz=96, R=20.0)  # fields of 50 MB
    g = iblb.Simulation.from_workload(wl, storage=iblb.FP32_DEV)
    g.step(2)
    g.nodal_forces()
    before = free_bytes()
    g.fields()
    assert free_bytes() == before
    g.close()


def test_batch_read_keeps_nothing():
    import torch
    torch.cuda.init()
    wl = small_3d(n=128, nz=96, R=20.0)
    b = iblb.Batch(wl.lattice, iblb.FP32_DEV, 1 << 30, max_slots=2)
    slot = b.admit_workload(wl, n_steps=4)
    b.run(4)
    b.sync()
    before = free_bytes()
    b.fields(slot)
    assert free_bytes() == before
    b.close()
