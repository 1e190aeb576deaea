"""The edge-tail render (k_render_mixed), which serves models with a width below 1 px, against the
oracle: both tail rationals (the widest PSF within 2.12 px or not) at every window size, several window
sizes in one model (the fused merge counts a tile's items across launches), and coefficient updates that
cross 1 px and 2.12 px both ways.  One slice is narrow, the others as wide as the case says; the kernel
that ran is named by its timing."""
import numpy as np
import pytest

import oracle
from paper_2008_05858_gb300 import workloads as W
from tests.framecompare import compare, tie_boxes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def renderer():
    from paper_2008_05858_gb300.binding import Renderer

    r = Renderer(0, kernel_timing=1)
    yield r
    r.close()


def _model(seed, hi, **kw):
    w = W.small_config(seed=seed, sigma_range=(1.2, hi), **{**dict(n_lambda=90, n_slit=12), **kw})
    s = w.model.slices[0]
    s.sigma_x, s.sigma_y = np.array([0.9, 0.0, 0.0]), np.array([hi, 0.0, 0.0])
    return w


def _check(renderer, mid, sids, w, kernel, launches=1):
    from paper_2008_05858_gb300.binding import e2e_kernel_times

    got = renderer.render(mid, sids, "mixed", "f32")
    torch.cuda.synchronize()
    names = [n for n, _ in e2e_kernel_times(renderer.ctx)]
    assert names == [kernel] * launches + (["merge"] if kernel != "render_mixed" else [])
    m = renderer.models[mid]
    for g, o, t in zip(got, oracle.render(m, w.flux_for), tie_boxes(m, w.flux_for)):
        rep = compare(g.double().cpu().numpy(), o, ties=t)
        assert rep.ok, str(rep)


@pytest.mark.parametrize("K", [1, 3, 5, 7, 9, 11, 13, 15])
@pytest.mark.parametrize("hi", [1.9, 2.6])
def test_both_rationals(renderer, K, hi):
    w = _model(500 + K, hi, K=K)
    mid = renderer.load_model(w.model)
    try:
        _check(renderer, mid, renderer.load_spectra(w), w, "render_mixed")
    finally:
        renderer.unload_model(mid)


@pytest.mark.parametrize("hi", [1.9, 2.6])
def test_fused_merge_across_launches(renderer, hi):
    w = _model(520, hi, orders=3, trace_pitch=6.0, height=200)
    for i, s in enumerate(w.model.slices):
        s.K = (7, 11, 9)[i % 3]
    mid = renderer.load_model(w.model)
    try:
        _check(renderer, mid, renderer.load_spectra(w), w, "render_mixed", 3)
    finally:
        renderer.unload_model(mid)


def test_updates_across_the_widths(renderer):
    w = W.small_config(seed=530, n_lambda=150, n_slit=12, sigma_range=(1.3, 1.9))
    mid = renderer.load_model(w.model)
    sids = renderer.load_spectra(w)
    cx, cy, sx, sy = renderer.params(mid)
    narrow = np.array(sx)
    narrow[0:3] = [0.8, 0.0, 0.0]
    try:
        for nx, ny, kernel in ((sx, sy, "render_poly"), (narrow, sy, "render_mixed"), (narrow, 1.6 * sy, "render_mixed"),
                               (narrow, sy, "render_mixed"), (1.6 * sx, 1.6 * sy, "render_poly"), (sx, sy, "render_poly")):
            renderer.update(mid, cx, cy, nx, ny)
            _check(renderer, mid, sids, w, kernel)
    finally:
        renderer.unload_model(mid)


def test_update_widens_a_narrow_model(renderer):
    # loaded without the polynomial tables: the first wide update allocates them
    w = W.small_config(seed=531, n_lambda=150, n_slit=12, sigma_range=(0.7, 0.95))
    mid = renderer.load_model(w.model)
    sids = renderer.load_spectra(w)
    cx, cy, sx, sy = renderer.params(mid)
    try:
        for f, kernel in ((1.0, "render_mixed"), (1.8, "render_poly"), (1.0, "render_mixed"), (2.0, "render_poly")):
            renderer.update(mid, cx, cy, f * sx, f * sy)
            _check(renderer, mid, sids, w, kernel)
    finally:
        renderer.unload_model(mid)
