"""The strip forward on pixels of unequal sides: up to an aspect of 8 against the
FP64 oracle (relative L2 1e-5, the projector tests' tolerance); beyond, where
its windows would not be safe, the rays go one by one whatever the mode."""
import math

import numpy as np
import pytest

from _helpers import rel_l2, to_dev, to_host
from synth import FAN2D, PAR2D, Geometry

pytestmark = pytest.mark.gpu


def _geometry(kind, dx, dy):
    size = 40 * max(dx, dy)
    return Geometry(kind, 40, 37, 1, dx, dy, 1.0, 21, 0.1, 2 * math.pi, 67, 1, 1.4 * size / 67 * (2 if kind == FAN2D else 1),
                    1.0, 2 * size, 4 * size)


@pytest.mark.parametrize("kind", [PAR2D, FAN2D])
@pytest.mark.parametrize("aspect", [1.0, 3.0, 8.0, 8.1, 40.0])
def test_unequal_pixels(oracle_lib, kind, aspect):
    import paper_2010_01371_gb300 as psps
    for dx, dy in ((aspect, 1.0), (1.0, aspect)):
        g = _geometry(kind, dx, dy)
        x = np.random.default_rng(2).random((2,) + g.image_shape)
        plan = psps.Plan(g)
        plan.set_projector("strip")
        got = to_host(psps.mbir_project(plan, to_dev(x)))
        assert rel_l2(got, oracle_lib.Projector(g).project(x)) < 1e-5
        plan.set_projector("ray")
        if aspect > 8.0:
            assert np.array_equal(got, to_host(psps.mbir_project(plan, to_dev(x))))
