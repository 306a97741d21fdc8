"""Cone scans of few detector rows or few voxel layers: both sides of the lines
between the column kernels and the general ones against the FP64 oracle
(relative L2 1e-5, the projector tests' tolerance), and that such a scan costs
accordingly."""
import math

import numpy as np
import pytest

import synth
from _helpers import rel_l2, to_dev, to_host
from synth import Geometry

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _g(nx, nz, views, nu, nv, dv=1.0):
    return Geometry(synth.CONE3D, nx, nx - 1, nz, 0.5, 0.5, 0.5, views, 0.17, 2 * math.pi, nu, nv, 1.0, dv, 600.0, 1200.0)


# rows, layers: around 4, 8 and 12 rows or layers (transpose), 17 and 32 rows that meet the volume (forward), layers
# in two groups of 32, and rows that mostly miss the volume
@pytest.mark.parametrize("nv,nz", [(1, 1), (3, 9), (4, 4), (8, 7), (11, 12), (12, 11), (16, 16), (17, 18), (31, 33),
                                   (33, 31), (24, 70), (40, 3)])
def test_few_rows_against_oracle(oracle_lib, nv, nz):
    import paper_2010_01371_gb300 as psps
    for nx, nu in ((19, 33), (130, 140)):
        g = _g(nx, nz, 7, nu, nv)
        A = oracle_lib.Projector(g)
        rng = np.random.default_rng(nv * 100 + nz)
        plan = psps.Plan(g)
        for n in (1, 2, 3):
            x, s = rng.random((n,) + g.image_shape), rng.random((n, g.n_rays))
            assert rel_l2(to_host(psps.mbir_project(plan, to_dev(x))), A.project(x)) < TOL, (nx, n)
            assert rel_l2(to_host(psps.mbir_backproject(plan, to_dev(s))), A.backproject(s)) < TOL, (nx, n)


def _ms(call):
    import torch
    for _ in range(3):
        call()
    t = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b))
    return sorted(t)[4]


@pytest.mark.parametrize("n", [1, 2])
def test_one_row_costs_less_than_many(n):
    """One row and layer of a 256 x 256 scan do at most a third of the forward time and 0.7 of the transpose time of
    32 rows and layers (a thirtieth and a seventh of the work)."""
    import torch
    import paper_2010_01371_gb300 as psps
    ms = {}
    for rows in (1, 32):
        g = Geometry(synth.CONE3D, 256, 256, rows, 0.5, 0.5, 0.5, 180, 0.0, 2 * math.pi, 512, rows, 0.8, 0.8, 600.0, 1200.0)
        plan = psps.Plan(g)
        x, l = torch.rand((n,) + g.image_shape, device="cuda"), torch.rand((n, g.n_rays), device="cuda")
        ms[rows] = _ms(lambda: psps.mbir_project(plan, x, l)), _ms(lambda: psps.mbir_backproject(plan, l, x))
    assert ms[1][0] < ms[32][0] / 3, ms
    assert ms[1][1] < 0.7 * ms[32][1], ms


def test_one_row_plan_memory():
    """A one-row plan holds 24 bytes of ray table and 16 of weighted sinogram per ray, not the column transpose's zero
    rows (16 rows of 16 bytes) around every column."""
    import torch
    import paper_2010_01371_gb300 as psps
    g = _g(64, 1, 1500, 4000, 1)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    plan = psps.Plan(g)
    used = free - torch.cuda.mem_get_info()[0]
    assert plan.n_rays == g.n_rays
    assert used < 80 * g.n_rays, used / g.n_rays
