"""Binary16 runs with the ordered spread are functions of their inputs, and the
stochastic rounding makes another trajectory of any change of a last bit (the
velocity then differs by about 1e-4).  These runs hold every kernel on their way
to the bits that they have always had: the digests are of populations and node
positions as first recorded on this architecture."""
import hashlib

import numpy as np
import pytest

from helpers import small_2d, small_3d
from paper_2604_17463_gb300 import iblb

pytestmark = pytest.mark.gpu

STEPS = 40
WALLS = dict(wall_u_lo=(-0.01, 0.0, 0.0), wall_u_hi=(0.015, 0.0, 0.0))
# 32 and 64 are widths that the pipelined kernel takes, 30 and 51 are not
SINGLE = {
    "2d_64": (("2d", 64, 40), {}, None),
    "2d_51": (("2d", 51, 40), {}, None),
    "2d_51_elastic": (("2d", 51, 40), dict(shear_modulus=1e-3), None),
    "2d_51_ratio": (("2d", 51, 40), dict(tau_out=0.7), None),
    "2d_64_ratio": (("2d", 64, 40), dict(tau_out=0.7), None),
    "3d_30": (("3d", 30, 22), {}, None),
    "3d_32": (("3d", 32, 22), {}, None),
    "3d_30_elastic": (("3d", 30, 22), dict(shear_modulus=1e-3), None),
    "3d_30_ratio": (("3d", 30, 22), dict(tau_out=0.7), None),
    "3d_32_ratio": (("3d", 32, 22), dict(tau_out=0.7), None),
    "3d_32_walls": (("3d", 32, 22), WALLS, None),
    "3d_30_overlapped": (("3d", 30, 22), {}, dict(variant=0, step_overlap=1)),
    "3d_30_overlapped_rows": (("3d", 30, 22), {}, dict(variant=3, step_overlap=1)),
    "3d_32_overlapped_rows": (("3d", 32, 22), {}, dict(variant=3, step_overlap=1)),
    "3d_32_overlapped_pipelined": (("3d", 32, 22), {}, dict(variant=1, step_overlap=1)),
    "3d_30_pairs": (("3d", 30, 22), {}, dict(variant=2)),
    "3d_30_grouped": (("3d", 30, 22), {}, dict(variant=0, ib_grouped=1)),
}
BATCH = {"batch_2d": (("2d", 64, 40), ("2d", 51, 33)), "batch_3d": (("3d", 32, 22), ("3d", 25, 23))}


def workload(kind, n, m):
    wl = small_2d(nx=n, ny=m) if kind == "2d" else small_3d(n=n, nz=m, R=7.0, level=3)
    # the same nodes whatever the host's sine rounds to
    wl.nodes = np.round(wl.nodes * 2.0 ** 20) / 2.0 ** 20
    return wl


def sha(*arrays):
    h = hashlib.sha256()
    for a in arrays:
        h.update(np.ascontiguousarray(a, dtype=np.float64).tobytes())
    return h.hexdigest()[:16]


def digest(name):
    if name in BATCH:
        wls = [workload(*w) for w in BATCH[name]]
        b = iblb.Batch(wls[0].lattice, iblb.FP16_DEV, 1 << 28, max_slots=2)
        slots = [b.admit_workload(w, n_steps=STEPS, deterministic_spread=True) for w in wls]
        b.run(STEPS)
        out = [x for s in slots for x in b.fields(s)]
        b.close()
        return sha(*out)
    which, over, tuning = SINGLE[name]
    g = iblb.Simulation.from_workload(workload(*which), storage=iblb.FP16_DEV, deterministic_spread=True, **over)
    if tuning:
        g.set_tuning(**tuning)
    g.step(STEPS)
    out = g.populations(), g.fields()[2]
    g.close()
    return sha(*out)


DIGESTS = {
    "2d_64": "bbcdc876ffbcdb10",
    "2d_51": "0d3a640c4af45691",
    "2d_51_elastic": "b09db00d85e3393b",
    "2d_51_ratio": "120f108a763c3005",
    "2d_64_ratio": "fdae9f5d7f85a0a6",
    "3d_30": "d34c387723f130c0",
    "3d_32": "b593f0ee10ba16e3",
    "3d_30_elastic": "2db269e48aadd417",
    "3d_30_ratio": "aa47379401c84596",
    "3d_32_ratio": "a2d54c2d7319a899",
    "3d_32_walls": "119d465072bf4422",
    "3d_30_overlapped": "d34c387723f130c0",
    "3d_30_overlapped_rows": "3e244a09b6069f84",
    "3d_32_overlapped_rows": "d4d83e81bf250ae7",
    "3d_32_overlapped_pipelined": "b901bdbcf2c99100",
    "3d_30_pairs": "bbe6eb6c86b0b595",
    "3d_30_grouped": "d34c387723f130c0",
    "batch_2d": "59efb2c97553d34a",
    "batch_3d": "8a793e21512463b8",
}


@pytest.mark.parametrize("name", list(SINGLE) + list(BATCH))
def test_ordered_binary16_run_keeps_its_bits(name):
    assert digest(name) == DIGESTS[name]
