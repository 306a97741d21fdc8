"""The spectral model's packed energy loops: odd ray counts (a thread's second
ray missing), every material and channel bound, and spectra whose channels see
different energy ranges, against the FP64 oracle.

Tolerance: 1e-5 relative L2, as every model test (FP32 exponents of at most 30
carry 30 x 2^-24 = 2e-6)."""
import numpy as np
import pytest

from _helpers import rel_l2, to_dev, to_host

pytestmark = pytest.mark.gpu

TOL = 1e-5


def _spectrum(kind, ne, nm, nc, rng):
    Q = rng.uniform(0.005, 0.03, (ne, nm))
    S = rng.uniform(10.0, 1000.0, (nc, ne))
    if kind == "disjoint":                       # photon counting: one channel per energy, some energies unseen
        S *= (np.arange(ne) * nc // ne)[None, :] == np.arange(nc)[:, None]
        S[:, :: 7] = 0.0
    elif kind == "nested":                       # tube voltages: channel c ends at its own energy
        S *= np.arange(ne)[None, :] < (np.arange(1, nc + 1) * ne // nc)[:, None]
    elif kind == "scattered":                    # more ranges than the table of ranges holds
        S *= rng.random((nc, ne)) < 0.5
    return Q, S


@pytest.mark.parametrize("kind", ["full", "disjoint", "nested", "scattered"])
@pytest.mark.parametrize("nm,nc,n", [(1, 1, 1), (1, 3, 257), (2, 2, 511), (3, 4, 70001), (4, 8, 1023)])
def test_model_ranges(kind, nm, nc, n):
    import paper_2010_01371_gb300 as psps
    from oracle import model
    rng = np.random.default_rng(nm * 100 + nc)
    ne = 1 if nc == 1 else 37
    Q, S = _spectrum(kind if ne > 1 else "full", ne, nm, nc, rng)
    l = rng.uniform(-1.0, 200.0 / nm, (nm, n)).astype(np.float32).astype(np.float64)
    y = rng.poisson(S @ np.exp(-(Q @ (0.9 * l)))).astype(np.float64)
    spec = psps.Spectrum(Q, S)
    ld, yd = to_dev(l), to_dev(y)
    g, obj = psps.mbmd_gradient(None, spec, ld, yd)
    assert rel_l2(to_host(g), model.data_grad_l(Q, S, l, y)) < TOL
    want = model.data_objective(Q, S, l, y)
    assert abs(float(obj) - want) <= TOL * want
    k = psps.mbmd_curvature(None, spec, ld, yd)
    assert rel_l2(to_host(k), model.curvature_numerator(Q, S, l, y, np.ones_like(l))) < TOL
