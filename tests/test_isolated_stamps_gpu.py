"""Single stamps, each alone on its part of the frame, at random sub-pixel offsets: nothing averages
a stamp's own rounding, so every pixel of the window has to meet the bound by itself, the wings of the
narrowest PSFs included.  The weight sits on one point of a slit that the mapping bends and tilts."""
import numpy as np
import pytest

import oracle
from paper_2008_05858_gb300 import workloads as W
from tests.framecompare import compare

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CELL = 40


def isolated(seed, sigma, K, psf=W.PSF_SEPARABLE, grid=24, n_slit=16, points=1, theta_deg=0.0):
    """grid x grid slices of one sample, widths within sigma .. 1.3 sigma, `points` slit points lit."""
    rng = np.random.default_rng(seed)
    d, nc = 5, W.n_coeffs(5)
    slices, flux = [], {}
    for n in range(grid * grid):
        cx, cy = np.zeros(nc), np.zeros(nc)
        for t in range(2, d + 1):
            for b in range(t + 1):
                cx[W.coeff_index(t - b, b)], cy[W.coeff_index(t - b, b)] = rng.uniform(-1, 1, 2) * 2.0 ** -t
        cx[W.coeff_index(0, 1)], cy[W.coeff_index(0, 1)] = rng.uniform(-1, 1), 4.0
        k = int(rng.integers(n_slit - points + 1))
        s = (2 * k + points - n_slit) / n_slit
        for c, cell in ((cx, n % grid), (cy, n // grid)):
            off = sum(c[W.coeff_index(0, b)] * s ** b for b in range(1, d + 1))
            c[0] = (cell + 0.5) * CELL + rng.uniform(-0.5, 0.5) - off
        u = np.zeros(n_slit)
        u[k:k + points] = rng.uniform(0.5, 1.0, points)
        sx, sy = sigma * rng.uniform(1.0, 1.3, 2)
        slices.append(W.OrderSlice(
            detector=0, order=n + 1, fiber=0, slice=0, degree=d, K=K, n_lambda=1, n_slit=n_slit, lambda_lo=5000.0,
            lambda_hi=5001.0, cx=cx, cy=cy, sigma_x=np.array([sx, 0.0, 0.0]), sigma_y=np.array([sy, 0.0, 0.0]),
            theta=np.deg2rad(theta_deg) * rng.uniform(-1, 1), slit_weights=u))
        flux[n + 1] = np.array([1000.0])
    m = W.OpticalModel([(grid * CELL, grid * CELL)], slices, psf)
    return W.Workload("isolated", m, {0: W.Spectrum(0, flux)}, "f32", "mixed")


def render(w):
    from paper_2008_05858_gb300.binding import Renderer

    r = Renderer(0)
    try:
        out = r.render(r.load_model(w.model), r.load_spectra(w), "mixed", "f32")
        torch.cuda.synchronize()
        return out[0].double().cpu().numpy()
    finally:
        r.close()


@pytest.mark.parametrize("K", [7, 9, 11, 13, 15])
@pytest.mark.parametrize("sigma", [1.0, 1.05, 1.1, 1.2, 1.3, 1.5, 1.8])
def test_separable(sigma, K):
    w = isolated(int(100 * sigma) + K, sigma, K)
    rep = compare(render(w), oracle.render_workload(w)[0])
    print(rep)
    assert rep.ok, str(rep)
