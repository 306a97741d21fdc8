"""The one-kernel middle of a cross-material Fourier apply on both sides of its
lines (two and four columns per CTA, separate passes), against FP64 FFTs
(relative L2 1e-5, the preconditioner tests' tolerance), and its cost on large
images."""
import math

import numpy as np
import pytest

from _helpers import rel_l2, to_dev, to_host
from synth import PAR2D, Geometry

pytestmark = pytest.mark.gpu


def _apply(nx, ny, nm, seed):
    """(library apply of M, FP64 result) for smooth spectra and unit M0 blocks."""
    import paper_2010_01371_gb300 as psps
    rng = np.random.default_rng(seed)
    r = np.hypot(np.fft.fftfreq(ny)[:, None], np.fft.fftfreq(nx)[None, :]).astype(np.float32).astype(np.float64)
    lam = np.zeros((nm, nm, ny, nx))
    for a in range(nm):
        lam[a, a] = (1.0 + 0.5 * a) / (0.1 + r)
        for b in range(a):
            lam[a, b] = lam[b, a] = 0.15 / (0.3 + r)
    v = rng.standard_normal((nm, ny, nx))
    plan = psps.Plan(Geometry(PAR2D, nx, ny, 1, 1.0, 1.0, 1.0, 3, 0.0, math.pi, 4, 1, 1.0, 1.0))
    spec = psps.Spectrum(np.ones((1, nm)), np.ones((1, 1)))
    blocks = np.repeat(np.eye(nm)[:, :, None], nx * ny, 2)
    pc = psps.Precond(plan, spec, "block_fourier", lam=to_dev(lam.reshape(nm, nm, -1)), blocks=to_dev(blocks))
    w, V = np.linalg.eigh(np.moveaxis(lam, (0, 1), (2, 3)))
    L = np.einsum("yxik,yxk,yxjk->ijyx", V, w ** -0.5, V)
    want = np.fft.ifft2(np.einsum("ijyx,jyx->iyx", L, np.fft.fft2(v))).real
    vd = to_dev(v)
    return (lambda: psps.psps_precondition(pc, "M", vd)), want


# two columns below 608 wide, four above, separate passes where they take too much shared memory
@pytest.mark.parametrize("nx,ny,nm", [(7, 630, 2), (600, 700, 4), (600, 14, 4), (625, 30, 2), (630, 640, 2), (630, 64, 4),
                                      (640, 625, 3), (700, 640, 4), (768, 1000, 2), (64, 1024, 4), (512, 1024, 3)])
def test_columns_per_block(nx, ny, nm):
    call, want = _apply(nx, ny, nm, nx + ny)
    assert rel_l2(to_host(call()), want) < 1e-5


def test_cost_of_four_materials():
    """Four materials of 700 x 700 are at most 1.75 times two (twice the work, in larger launches)."""
    import torch
    ms = {}
    for nm in (2, 4):
        call, _ = _apply(700, 700, nm, 1)
        for _ in range(5):
            call()
        t = []
        for _ in range(15):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            call()
            b.record()
            torch.cuda.synchronize()
            t.append(a.elapsed_time(b))
        ms[nm] = sorted(t)[7]
    assert ms[4] <= 1.75 * ms[2], ms
