"""What a scan of many rays runs by default: strips for the images they pay for,
one thread per ray for smaller ones (bitwise what those modes give), and the
mode that was chosen once one is."""
import math

import numpy as np
import pytest

from _helpers import to_dev, to_host
from synth import FAN2D, Geometry

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(64, 64), (191, 192), (192, 192), (351, 352), (352, 352)])
def test_default_forward(nx, ny):
    import paper_2010_01371_gb300 as psps
    g = Geometry(FAN2D, nx, ny, 1, 0.5, 0.5, 1.0, 620, 0.0, 2 * math.pi, 512, 1, nx / 512 * 1.6, 1.0, 2.0 * nx, 4.0 * nx)
    x = np.random.default_rng(1).random((6,) + g.image_shape).astype(np.float32)
    default, ray, strip = (psps.Plan(g) for _ in range(3))
    ray.set_projector("ray")
    strip.set_projector("strip")
    for n in (1, 2, 3, 4, 6):
        d, r, s = (to_host(psps.mbir_project(p, to_dev(x[:n]))) for p in (default, ray, strip))
        for m0 in range(0, n, 4):            # groups of four images and the rest
            k = min(4, n - m0)
            pays = nx * ny >= (352 if k in (1, 4) else 192) ** 2
            q = slice(m0, m0 + k)
            assert np.array_equal(d[q], (s if pays else r)[q]), (n, m0)
            assert not np.array_equal(r[q], s[q])
    default.set_projector("strip")
    assert np.array_equal(to_host(psps.mbir_project(default, to_dev(x[:1]))), to_host(psps.mbir_project(strip, to_dev(x[:1]))))
