"""The fixed-point tile scatter on the plans that run it by default (rays that
the z axis drives): signed data at both tile depths, a NaN, and the low words of
the gradient channels."""
import math

import numpy as np
import pytest

import synth
from _helpers import rel_l2, to_dev, to_host
from synth import Geometry

pytestmark = pytest.mark.gpu

# detector half-height above sdd / sqrt 2; the second with more than one tile along every axis
GEOMS = {
    "small": Geometry(synth.CONE3D, 14, 12, 30, 1.0, 1.0, 1.0, 9, 0.17, 2 * math.pi, 26, 60, 1.6, 2.2, 32.0, 45.0),
    "tiles": Geometry(synth.CONE3D, 25, 19, 35, 0.8, 0.9, 0.7, 13, 0.4, 2 * math.pi, 40, 72, 1.4, 1.6, 30.0, 52.0),
}


def _kernels(call):
    """Names of the kernels of one call (empty where the profiler records none)."""
    import torch
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return [e.key for e in prof.key_averages()]


@pytest.mark.parametrize("depth", [16, 8])
@pytest.mark.parametrize("name", list(GEOMS))
def test_signed_data(oracle_lib, name, depth):
    """Five channels over four decades of scale: 1e-5 relative L2 of the oracle, every voxel within 3e-6 of the
    channel's largest of the FP32 gather (a term carries at most half a unit of max |w s| 2^-22), bitwise repeatable."""
    import torch
    import paper_2010_01371_gb300 as psps
    g = GEOMS[name]
    s = np.random.default_rng(18).standard_normal((5, g.n_rays)) * np.array([1.0, 1e-2, 1e2, 3.0, 0.5])[:, None]
    plan, gather = psps.Plan(g), psps.Plan(g)
    plan.set_cone_tile(depth)
    gather.set_backprojector("gather")
    names = _kernels(lambda: psps.mbir_backproject(plan, to_dev(s)))
    assert not names or any("back_cone_tile" in k for k in names), names
    a = to_host(psps.mbir_backproject(plan, to_dev(s)))
    assert np.array_equal(a, to_host(psps.mbir_backproject(plan, to_dev(s))))
    z = torch.zeros((5,) + g.image_shape, device="cuda", dtype=torch.float32)
    assert np.array_equal(a, to_host(psps.mbir_backproject(plan, to_dev(s), z, accumulate=True)))
    want, ref = oracle_lib.Projector(g).backproject(s), to_host(psps.mbir_backproject(gather, to_dev(s)))
    for c in range(5):
        assert rel_l2(a[c], want[c]) < 1e-5
        assert np.abs(a[c] - ref[c]).max() <= 3e-6 * np.abs(ref[c]).max()
    s[1, 11] = np.nan
    b = to_host(psps.mbir_backproject(plan, to_dev(s)))
    assert np.isnan(b[1]).all() and np.array_equal(np.delete(b, 1, 0), np.delete(a, 1, 0))


@pytest.mark.parametrize("depth", [16, 8])
@pytest.mark.parametrize("name", list(GEOMS))
def test_gradient_low_words(oracle_lib, name, depth):
    """One ray without counts has a numerator some 1e5 times the others', which sets the grid of its channel: the
    voxels it does not reach keep their gradient to N units of M 2^-32 (the grid M 2^-20 at most, its low words 2^-12
    of it), N the terms of a voxel."""
    import paper_2010_01371_gb300 as psps
    from oracle import model
    g = GEOMS[name]
    A = oracle_lib.Projector(g)
    rng = np.random.default_rng(2)
    x = rng.random((1,) + g.image_shape) * 0.05
    Q, S = np.ones((1, 1)), np.full((1, 1), 1e4)
    x = x.astype(np.float32).astype(np.float64)
    l = A.project(x)
    y = rng.poisson(S @ np.exp(-Q @ l)).astype(np.float64)
    hot = g.n_rays // 2 + 3
    y[0, hot] = 0.0
    spec, plan = psps.Spectrum(Q, S), psps.Plan(g)
    plan.set_cone_tile(depth)
    got = to_host(psps.mbmd_gradient(plan, spec, to_dev(x), to_dev(y), with_objective=False)[0])
    num = model.data_grad_l(Q, S, l, y)
    one = np.zeros((1, g.n_rays))
    one[0, hot] = 1.0
    away = A.backproject(one) == 0.0
    assert abs(num[0, hot]) > 2e3 * np.median(np.abs(num)) and away.any()
    want = A.backproject(num)
    terms = float(A.backproject(np.ones((1, g.n_rays))).max()) * 4.0        # mean weight of a term above a quarter
    unit = float(np.abs(num).max()) * 1.75 * 2.0 ** -32
    other = np.abs(np.delete(num, hot, 1)).max()
    err = np.abs(got - want)[away].max()
    assert err <= terms * unit + 1e-5 * other * terms ** 0.5, (err, terms * unit)
