"""Edges of the strip forward and of the one-CTA Haar apply, against the FP64
oracle (relative L2 1e-5, the tolerance of the projector and preconditioner
apply tests)."""
import math

import numpy as np
import pytest

from _helpers import rel_l2, to_dev, to_host
from synth import FAN2D, PAR2D, Geometry

pytestmark = pytest.mark.gpu

TOL = 1e-5

GEOMS = {
    "coarse_bins": Geometry(PAR2D, 301, 290, 1, 0.5, 0.5, 1.0, 23, 0.1, math.pi, 40, 1, 6.0, 1.0),   # windows above kSH
    "wide_fan": Geometry(FAN2D, 40, 37, 1, 1.0, 1.0, 1.0, 13, 0.2, 2 * math.pi, 70, 1, 3.0, 1.0, 40.0, 60.0),
    "two_groups": Geometry(PAR2D, 530, 21, 1, 1.0, 1.0, 1.0, 11, 0.05, math.pi, 97, 1, 1.0, 1.0),    # 17 strips of 32
    "one_bin": Geometry(FAN2D, 33, 65, 1, 1.0, 0.9, 1.0, 9, 0.0, 2 * math.pi, 1, 1, 1.0, 1.0, 90.0, 180.0),
    "default_strips": Geometry(FAN2D, 70, 66, 1, 0.6, 0.6, 1.0, 999, 0.0, 2 * math.pi, 321, 1, 0.3, 1.0, 90.0, 180.0),
}


@pytest.mark.parametrize("name", list(GEOMS))
@pytest.mark.parametrize("nm", [1, 2, 3, 4])
def test_strip_edges(oracle_lib, name, nm):
    import torch
    import paper_2010_01371_gb300 as psps
    g = GEOMS[name]
    x = np.random.default_rng(31).random((nm,) + g.image_shape)
    want = oracle_lib.Projector(g).project(x)
    plan = psps.Plan(g)
    assert (plan.tuning()["forward"] == "strip") == (name == "default_strips")
    off = torch.empty(x.size + 1, device="cuda")[1:].view(x.shape)     # rows that no 16-byte copy can start on
    off.copy_(to_dev(x))
    for sb in (32, 64):
        plan.set_projector("strip")
        plan.set_strip_bins(sb)
        assert rel_l2(to_host(psps.mbir_project(plan, to_dev(x))), want) < TOL
        assert rel_l2(to_host(psps.mbir_project(plan, off)), want) < TOL


@pytest.mark.parametrize("n", [2, 8, 32, 64, 128])
@pytest.mark.parametrize("sides", [1, 2])
def test_haar_apply_sizes(n, sides):
    import paper_2010_01371_gb300 as psps
    from oracle import precond
    rng = np.random.default_rng(n)
    lam, m0, v = rng.uniform(0.5, 4.0, (n, n)), rng.uniform(0.5, 2.0, (n, n)), rng.standard_normal((1, n, n))
    plan = psps.Plan(Geometry(PAR2D, n, n, 1, 1.0, 1.0, 1.0, 3, 0.0, math.pi, 4, 1, 1.0, 1.0))
    spec = psps.Spectrum(np.ones((1, 1)), np.ones((1, 1)))
    pc = psps.Precond(plan, spec, "haar", lam=to_dev(lam), m0=to_dev(m0), sides=sides)
    P = precond.Haar(lam, m0, sides)
    for op in ("M", "MT", "absM", "absMT"):
        assert rel_l2(to_host(psps.psps_precondition(pc, op, to_dev(v))), getattr(P, op)(v)) < TOL, op
