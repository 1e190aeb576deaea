"""Separable models that the polynomial kernel must not cost what the edge tails had: a work item whose
box leaves no room for its exchange renders from the tails, at load and after an update, and back."""
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


def _check(renderer, mid, sids, w, kernel):
    from paper_2008_05858_gb300.binding import e2e_kernel_times

    got = renderer.render(mid, sids, "mixed", "f32")
    torch.cuda.synchronize()
    assert kernel in [n for n, _ in e2e_kernel_times(renderer.ctx)]
    m = renderer.models[mid]
    for g, o, t in zip(got, oracle.render(m, w.flux_for), tie_boxes(m, w.flux_for)):
        rep = compare(g.double().cpu().numpy(), o, ties=t)
        assert rep.ok, str(rep)


def test_box_too_large_for_the_polynomials(renderer):
    # one item of 32 samples x 16 slit points spans the 120 x 224 frame: 26,880 box pixels, 215 KB
    w = W.small_config(seed=61, width=120, height=224, orders=1, fibers=1, slices=1, n_lambda=32, n_slit=16)
    for s in w.model.slices:
        s.cy[W.coeff_index(0, 1)] = 130.0
    mid = renderer.load_model(w.model)
    sids = renderer.load_spectra(w)
    cx, cy, sx, sy = renderer.params(mid)
    flat = np.array(cy)
    flat[W.coeff_index(0, 1)] = 20.0
    try:
        _check(renderer, mid, sids, w, "render_mixed")
        renderer.update(mid, cx, flat, sx, sy)
        _check(renderer, mid, sids, w, "render_poly")
        renderer.update(mid, cx, cy, sx, sy)
        _check(renderer, mid, sids, w, "render_mixed")
    finally:
        renderer.unload_model(mid)
