"""Cone transpose with many detector rows per voxel layer (several passes of
rows), element by element against the FP64 oracle.

Bound: a term is a product of two hat functions whose arguments are FP32
coordinates of at most c = n / 2 voxels with about three roundings each, so it
errs by at most delta = 2 x 3 c 2^-24 (slopes one).  A voxel receives at most
N = views x columns x rows terms whose errors are independent: 8 sqrt(N) delta
w_max, plus 1e-6 of the sum for the FP32 additions.  A row left out or counted
twice is off by a whole term, up to w_max."""
import math

import numpy as np
import pytest

import synth
from _helpers import to_dev, to_host
from synth import Geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dv,rows", [(0.7, 8), (0.4, 14), (0.3, 19)])      # two, three and four passes of six rows
@pytest.mark.parametrize("nch", [2, 4])
def test_rows_of_neighbouring_passes_join(oracle_lib, dv, rows, nch):
    import paper_2010_01371_gb300 as psps
    g = Geometry(synth.CONE3D, 64, 64, 128, 1.0, 1.0, 1.0, 60, 0.0, 2 * math.pi, 128, 384, 1.6, dv, 600.0, 1200.0)
    s = np.random.default_rng(5).random((nch, g.n_rays)).astype(np.float32)
    got = to_host(psps.mbir_backproject(psps.Plan(g), to_dev(s)))
    A = oracle_lib.Projector(g)
    n_terms = g.n_views * 4 * rows                 # columns are at least 0.73 voxels apart
    tol = 8 * math.sqrt(n_terms) * 2 * 3 * 64 * 2.0 ** -24 * math.sqrt(2.0) * 1.05
    for c in range(nch if nch == 2 else 1):
        want = A.backproject(s[c:c + 1])[0]
        err = np.abs(got[c] - want)
        assert np.all(err <= tol + 1e-6 * want.max()), (float(err.max()), tol, int(np.sum(err > tol)))
