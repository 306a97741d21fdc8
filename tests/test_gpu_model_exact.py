"""Numerators whose every factor is a small integer over a power of two: FP32
holds each product exactly, so the per-ray gradient and curvature numerators of
a one-energy scan at l = 0 (transmission 1) have to be exact."""
import numpy as np
import pytest

from _helpers import to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("row", [0, 32])          # independent rays; rays coupled along detector rows (a trivial blur)
def test_one_energy_numerators_are_exact(row):
    import paper_2010_01371_gb300 as psps
    l, y = np.zeros((1, 96)), np.full((1, 96), 512.0)
    for k in range(1, 256, 3):
        Q = k / 256.0
        spec = psps.Spectrum(np.full((1, 1), Q), np.full((1, 1), 1024.0))
        if row:
            spec.set_blur((0.0, 1.0, 0.0), row)
        g, obj = psps.mbmd_gradient(None, spec, to_dev(l), to_dev(y))
        # r = 1024 - 512, w = 1 / 512, v = S w r = 1024
        assert np.all(to_host(g) == -1024.0 * Q) and float(obj) == 96 * 256.0
        # eta = S w S = 2048, rho = v - eta = -1024, c = 2 eta + rho = 3072
        assert np.all(to_host(psps.mbmd_curvature(None, spec, to_dev(l), to_dev(y))) == 3072.0 * Q * Q)
