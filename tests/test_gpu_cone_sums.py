"""Rounding of the cone transpose's sums over many views, against the FP64
oracle.

Positive data, 5760 views in one split: a voxel's value is the sum of a few
thousand terms of like size.  Their own errors (a few 2^-24 of a coordinate of
at most 200 voxels, 4e-5 of a term) are independent and average to below
1e-6 / sqrt(5760 / 2) = 2e-8 of the sum; the total is rounded to FP32 once,
2^-24 at most: relative L2 within 2^-24 + 2e-8 = 8e-8.  Adding group after
group of views to one FP32 number errs by 2^-25 sqrt(groups / 3), 2e-7 here."""
import math

import numpy as np
import pytest

import synth
from _helpers import to_dev, to_host
from synth import Geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nch", [2, 4])
def test_sum_over_many_views(oracle_lib, nch):
    import paper_2010_01371_gb300 as psps
    g = Geometry(synth.CONE3D, 384, 384, 12, 0.5, 0.5, 0.5, 5760, 0.0, 2 * math.pi, 16, 12, 4.0, 1.0, 600.0, 1200.0)
    s = np.random.default_rng(9).uniform(0.5, 1.5, (1, g.n_rays)).astype(np.float32)
    want = oracle_lib.Projector(g).backproject(s)[0]
    got = to_host(psps.mbir_backproject(psps.Plan(g), to_dev(np.repeat(s, nch, 0))))
    inner = want > 0.2 * want.max()
    for c in range(nch):
        e = np.linalg.norm((got[c] - want)[inner]) / np.linalg.norm(want[inner])
        assert e < 8e-8, e
