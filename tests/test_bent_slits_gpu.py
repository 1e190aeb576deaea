"""Single stamps at the ends of slits bent as far as the FP32 mapping takes them (1 px between a sample's
straight slit and the stamp) and tilted by up to 60 px: the rounding of the offset reaches the wings of the
narrowest PSFs first, and every pixel has to meet the bound.  Just beyond the limit the exact mapping serves."""
import numpy as np
import pytest

import oracle
from paper_2008_05858_gb300 import workloads as W
from tests.framecompare import compare
from tests.test_isolated_stamps_gpu import CELL, isolated, render

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def bent(seed, sigma, K, psf, bend, tilt, grid=24, n_slit=64):
    theta = 10.0 if psf == W.PSF_ELLIPTICAL else 0.0
    w = isolated(seed, sigma, K, psf=psf, grid=grid, n_slit=n_slit, theta_deg=theta)
    rng = np.random.default_rng(seed + 999)
    at = [W.coeff_index(0, b) for b in range(6)]
    for n, s in enumerate(w.model.slices):
        k = int(rng.choice([0, 1, 2, n_slit - 3, n_slit - 2, n_slit - 1]))
        s.slit_weights = np.where(np.arange(n_slit) == k, rng.uniform(0.5, 1.0), 0.0)
        t = (2 * k + 1 - n_slit) / n_slit
        for c, cell in ((s.cx, n % grid), (s.cy, n // grid)):
            c[:] = 0.0
            c[at[2:]] = rng.dirichlet(np.ones(4)) * bend * np.sign(t) ** np.arange(2, 6) * rng.choice([-1, 1])
            c[at[1]] = rng.uniform(-tilt, tilt)
            c[0] = (cell + 0.5) * CELL + rng.uniform(-0.5, 0.5) - sum(c[at[b]] * t ** b for b in range(1, 6))
    return w


@pytest.mark.parametrize("bend", [0.5, 0.999, 1.2])
@pytest.mark.parametrize("K", [11, 13])
@pytest.mark.parametrize("psf,sigma,tilt", [(W.PSF_SEPARABLE, 1.0, 60.0), (W.PSF_SEPARABLE, 1.1, 60.0),
                                            (W.PSF_ELLIPTICAL, 1.3, 4.0)])
def test_bent(psf, sigma, tilt, K, bend):
    w = bent(int(100 * sigma) + K, sigma, K, psf, bend, tilt)
    rep = compare(render(w), oracle.render_workload(w)[0])
    print(rep)
    assert rep.ok, str(rep)
