"""The elliptical render's tables along the slice, where their interpolation is worst: widths that
hardly change but are curved (their slope alone would allow nodes far apart), slices of fewer samples
than an interval, and coefficient updates that take a model from one kernel to the other and back.
Against the oracle, with the kernel that ran named by its timing."""
import numpy as np
import pytest

import oracle
from paper_2008_05858_gb300 import workloads as W
from tests.framecompare import compare

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    from paper_2008_05858_gb300.binding import Renderer

    r = Renderer(0, kernel_timing=1)
    yield r
    r.close()


def _model(n_lambda, c2, c1=0.0, c0=1.5):
    w = W.small_config(seed=460, psf=W.PSF_ELLIPTICAL, orders=1, fibers=1, slices=1, n_lambda=n_lambda, n_slit=5,
                       K=13, width=160, height=60)
    s = w.model.slices[0]
    s.theta = np.deg2rad(5.0)
    s.sigma_x, s.sigma_y = np.array([c0, c1, c2]), np.array([c0, -c1, c2])
    return w


def _check(renderer, mid, sids, model, w, kernel):
    from paper_2008_05858_gb300.binding import e2e_kernel_times

    got = renderer.render(mid, sids, "mixed", "f32")
    torch.cuda.synchronize()
    names = {n for n, _ in e2e_kernel_times(renderer.ctx)}
    assert names == {kernel, "merge"}
    for g, o in zip(got, oracle.render(model, w.flux_for)):
        rep = compare(g.double().cpu().numpy(), o)
        assert rep.ok, str(rep)


CASES = [(16, 3e-4, "render_ellip"), (32, 1e-2, "render_ellip"), (3000, 0.0, "render_moments"), (16, 0.0, "render_moments")]
CASES += [(3000, c2, "render_moments") for c2 in (3e-4, 1e-3, 2e-3, 5e-3, 1e-2, -1e-2)]


@pytest.mark.parametrize("n_lambda,c2,kernel", CASES)
def test_curved_widths(renderer, n_lambda, c2, kernel):
    w = _model(n_lambda, c2)
    mid = renderer.load_model(w.model)
    sids = renderer.load_spectra(w)
    try:
        _check(renderer, mid, sids, w.model, w, kernel)
    finally:
        renderer.unload_model(mid)


def test_updates_across_the_limits(renderer):
    w = _model(1500, 5e-3, c1=0.02)
    mid = renderer.load_model(w.model)
    sids = renderer.load_spectra(w)
    cx, cy, sx, sy = renderer.params(mid)
    try:
        # as loaded; narrower than the moments serve; varying too fast; as loaded; wider, steeper
        for f, kernel in ((lambda v: v, "render_moments"), (lambda v: 0.6 * v, "render_ellip"),
                          (lambda v: v + np.array([1.0, 0.6, 0.3]), "render_ellip"), (lambda v: v, "render_moments"),
                          (lambda v: 1.3 * v + np.array([0.0, 0.02, 0.0]), "render_moments")):
            nx, ny = (np.array([f(c) for c in np.asarray(v).reshape(-1, 3)]).reshape(np.shape(v)) for v in (sx, sy))
            renderer.update(mid, cx, cy, nx, ny)
            _check(renderer, mid, sids, renderer.models[mid], w, kernel)
    finally:
        renderer.unload_model(mid)
