"""Sums of the strip forward: rays through pixel centres along an image axis
sum whole numbers of up to 21 bits, whose partial sums of eight FP32 holds
exactly, with weight 1.  Every row's sum is small although its parts reach
2^28, so a compensated total of such partials is off by less than
2^-24 |sum| + n 2^-48 2^28 < 0.1."""
import numpy as np
import pytest

from _helpers import to_dev, to_host
from synth import PAR2D, Geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nm", [1, 2, 3, 4])
def test_cancelling_rows(nm):
    import paper_2010_01371_gb300 as psps
    n = 512
    g = Geometry(PAR2D, n, 64, 1, 1.0, 1.0, 1.0, 1, 0.0, 1.0, 64, 1, 1.0, 1.0)
    rng = np.random.default_rng(4)
    x = np.empty((nm, 64, n))
    x[:, :, : n // 2] = rng.integers(2 ** 20, 2 ** 21, (nm, 64, n // 2)) | 1
    x[:, :, n // 2:] = -rng.permuted(x[:, :, : n // 2], axis=2)
    x[:, :, -1] += rng.integers(0, 1000, (nm, 64))
    plan = psps.Plan(g)
    plan.set_projector("strip")
    got = to_host(psps.mbir_project(plan, to_dev(x)))
    assert np.abs(got - x.sum(2)).max() < 0.1
