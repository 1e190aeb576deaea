"""The rotated PSF's stamps and runs, each alone on its part of the frame: every pixel of a run's
window has to meet the bound by itself, also where all the run's stamps lie on one side of their pixel
and the wing opposite is what large terms leave over.  One stamp; 100 stamps within a third of a pixel;
the same with weights over four decades."""
import numpy as np
import pytest

import oracle
from paper_2008_05858_gb300 import workloads as W
from tests.framecompare import compare
from tests.test_isolated_stamps_gpu import isolated, render

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [5, 9, 11, 13])
@pytest.mark.parametrize("sigma", [1.0, 1.2, 1.25, 1.3, 1.4, 1.5])
def test_one_stamp(sigma, K):
    w = isolated(int(100 * sigma) + K, sigma, K, psf=W.PSF_ELLIPTICAL, theta_deg=10.0)
    rep = compare(render(w), oracle.render_workload(w)[0])
    print(rep)
    assert rep.ok, str(rep)


@pytest.mark.parametrize("decades", [0, 4])
@pytest.mark.parametrize("sigma", [1.0, 1.25, 1.3, 1.5])
def test_run_on_one_side(sigma, decades):
    w = isolated(int(1000 * sigma) + decades, sigma, 13, psf=W.PSF_ELLIPTICAL, theta_deg=10.0, grid=16, n_slit=2400,
                 points=100)
    rng = np.random.default_rng(5)
    for s in w.model.slices:
        s.slit_weights = s.slit_weights * 10.0 ** -rng.uniform(0, decades, len(s.slit_weights))
    rep = compare(render(w), oracle.render_workload(w)[0])
    print(rep)
    assert rep.ok, str(rep)


def test_narrow_slices_beside_wide_ones():
    # slices on either side of the moments' width limit, two window sizes: each renders by its own kernel
    from paper_2008_05858_gb300.binding import Renderer, e2e_kernel_times

    w = isolated(81, 1.0, 13, psf=W.PSF_ELLIPTICAL, theta_deg=10.0, grid=12, n_slit=40, points=7)
    for i, s in enumerate(w.model.slices):
        s.K = (13, 15, 9)[i % 3]
        if i % 2:
            s.sigma_x, s.sigma_y = 1.5 * s.sigma_x, 1.5 * s.sigma_y
    r = Renderer(0, kernel_timing=1)
    try:
        mid = r.load_model(w.model)
        sids = r.load_spectra(w)
        out = r.render(mid, sids, "mixed", "f32")
        torch.cuda.synchronize()
        names = [n for n, _ in e2e_kernel_times(r.ctx)]
        assert names.count("render_ellip") == 3 and names.count("render_moments") == 2 and names[-1] == "merge"
        rep = compare(out[0].double().cpu().numpy(), oracle.render_workload(w)[0])
        assert rep.ok, str(rep)
        host = r.render_host(mid, sids)
        assert np.array_equal(host[0].numpy(), out[0].cpu().numpy())
    finally:
        r.close()
