"""GPU kernels and dispatch rules at the sizes where they can go wrong, against the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
from tests import seeded
from tests.test_gpu_parity import L, perturbed, rel  # noqa: F401  (L: the module fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e30])
@pytest.mark.parametrize("q,dims,periodic", [
    (9, (128, 128, 1), 0),   # plain steps in CTAs of one row
    (9, (33, 301, 1), 1),    # of a few rows, a partial CTA at the end
    (9, (700, 303, 1), 2),   # whole CTAs
    (19, (33, 9, 17), 0), (19, (1, 2, 3), 0), (19, (40, 8, 24), 4)])
def test_fp64_pairwise_relaxation(L, q, dims, periodic, scale):  # noqa: F811
    """The FP64 relaxation, which adds the sensor's fractions over common denominators, at densities
    far from 1 too.  A step rounds each population a few times at 2^-53 of its size and K a few
    tens of times at 2^-53 of f / f^neq (about 50 here): 1e-14 and 1e-12 leave a margin of ten."""
    o = O.Oracle(q, *dims, tau=0.83, lid=(0.0, 0.0, 0.0), periodic=periodic)
    f = scale * perturbed(o, seed=17 + sum(dims), amp=0.02)
    lat = L.Lattice(q, *dims, 0.83, dtype=L.LBM_F64, lid=(0.0, 0.0), periodic=periodic)
    lat.set_populations(f)
    L.lbm_set_sensor_field(lat.h, 1)
    lat.step(3)  # two plain steps and a sensor step
    for _ in range(3):
        f, K, _, _ = o.step(f, sensor=True)
    assert rel(lat.populations(), f) <= 1e-14
    assert rel(lat.sensor_field(), K) <= 1e-12
    lat.close()
