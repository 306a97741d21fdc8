"""Cone projector over detector columns: the edges of its work split and the
geometries it leaves to the general kernels, against the FP64 oracle.

Tolerance: relative L2 1e-5 for projections and transposes of positive data,
the tolerance of every projector test (FP32 coordinates of at most 100 voxels
carry 100 x 2^-24 = 6e-6 of a voxel, and random signs average them)."""
import math

import numpy as np
import pytest

import synth
from _helpers import rel_l2, to_dev, to_host
from synth import Geometry

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _g(nx, ny, nz, views, nu, nv, du, dv, sid, sdd, vox=(1.0, 1.0, 1.0)):
    return Geometry(synth.CONE3D, nx, ny, nz, *vox, views, 0.17, 2 * math.pi, nu, nv, du, dv, sid, sdd)


GEOMS = {
    "rows_2": _g(17, 22, 33, 19, 24, 31, 3.2, 5.0, 90.0, 200.0),           # rows 1.8 voxels apart
    "rows_3": _g(20, 13, 64, 37, 40, 70, 1.9, 2.4, 110.0, 200.0),          # two rows of patches in y overhang
    "rows_4": _g(35, 30, 65, 33, 70, 97, 0.8, 0.8, 600.0, 1200.0, (0.5, 0.5, 0.5)),   # one z past a warp
    "rows_many": _g(18, 16, 20, 21, 110, 90, 0.5, 0.4, 60.0, 130.0, (0.9, 1.0, 1.2)),  # several passes of rows
    "one_voxel": _g(1, 1, 1, 6, 7, 5, 0.7, 0.6, 30.0, 60.0),
    "one_row": _g(12, 9, 5, 40, 30, 1, 1.0, 1.0, 60.0, 120.0),
    "one_column_one_view": _g(12, 9, 40, 1, 1, 80, 1.0, 1.0, 60.0, 120.0),
    "z_driven": _g(14, 12, 30, 9, 26, 60, 1.6, 2.2, 32.0, 45.0),           # detector half-height above sdd / sqrt 2
    "close_source": _g(16, 16, 12, 15, 30, 20, 1.1, 1.1, 12.0, 30.0),      # no bound on depth: the FP32 gather
}


@pytest.mark.parametrize("name", list(GEOMS))
@pytest.mark.parametrize("n", [1, 2, 4, 5])
def test_columns_against_oracle(oracle_lib, name, n):
    import paper_2010_01371_gb300 as psps
    g = GEOMS[name]
    A = oracle_lib.Projector(g)
    rng = np.random.default_rng(21)
    x, s = rng.random((n,) + g.image_shape), rng.random((n, g.n_rays))
    plan = psps.Plan(g)
    assert rel_l2(to_host(psps.mbir_project(plan, to_dev(x))), A.project(x)) < TOL
    want = A.backproject(s)
    got = psps.mbir_backproject(plan, to_dev(s))
    assert rel_l2(to_host(got), want) < TOL
    assert np.array_equal(to_host(got), to_host(psps.mbir_backproject(plan, to_dev(s))))
    base = to_dev(np.ones((n,) + g.image_shape))
    psps.mbir_backproject(plan, to_dev(s), base, accumulate=True)
    assert rel_l2(to_host(base), want + 1.0) < TOL
    if n == 2:                     # the alternatives read the table derived from the same columns
        for mode in ("gather", "split", "atomic"):
            plan.set_backprojector(mode)
            assert rel_l2(to_host(psps.mbir_backproject(plan, to_dev(s))), want) < TOL, mode
