"""The mass of FP32 and binary16 populations is their FP64 sum: on one cell,
whose sum needs no more than the 53 bits of FP64, it is the exact one."""
from fractions import Fraction

import numpy as np
import pytest

from paper_2604_17463_gb300 import iblb

pytestmark = pytest.mark.gpu

WEIGHTS = {9: [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, 19: [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12}


@pytest.mark.parametrize("Q", [9, 19])
@pytest.mark.parametrize("storage", [iblb.FP32_DEV, iblb.FP16_DEV])
def test_mass_of_a_cell_is_exact(Q, storage):
    s = iblb.Simulation(Q, 1, 1, 1, walls=False, wetting=False, storage=storage)
    w = np.array(WEIGHTS[Q])
    rng = np.random.default_rng(11)
    for _ in range(100):
        # deviations between 2^-26 and 1: multiples of 2^-49, their sum with the
        # 1 of the density below 2^5 - a weight can be added and taken off again
        # without losing a bit
        g = rng.choice([-1.0, 1.0], Q) * rng.uniform(1, 2, Q) * 2.0 ** rng.integers(-26, 0, Q)
        if storage == iblb.FP32_DEV:
            g = g.astype(np.float32).astype(np.float64)
        else:  # as stored: binary16 of the deviation times 2^16
            g = (g * 2.0 ** 14).astype(np.float16).astype(np.float64) / 2.0 ** 16
        s.set_populations((w + g).reshape(s.populations().shape))
        exact = 1 + sum(Fraction(float(x)) for x in g)
        assert Fraction(s.observables()["mass"]) == exact
    s.close()


@pytest.mark.parametrize("storage", [iblb.FP64, iblb.FP32_DEV])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_mass_of_a_diverged_cell(storage, bad):
    s = iblb.Simulation(9, 3, 2, 1, walls=False, wetting=False, storage=storage)
    f = s.populations()
    f[4, 0, 1, 1] = bad
    s.set_populations(f)
    assert np.array_equal(s.observables()["mass"], bad, equal_nan=True)
    s.close()
