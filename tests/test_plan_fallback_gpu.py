"""Separable models that the polynomial kernel must not cost what the edge tails had: a work item whose
box leaves no room for its exchange renders from the tails, at load and after an update, and back; so
does a model whose tables a nearly full device would not spare."""
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


def test_no_polynomials_on_a_full_device(renderer):
    # 320,000 samples: 41 MB of sample tables, 143 MB of polynomials, which a device with 0.4 GB left
    # does not spare (more than a quarter); an update there keeps the tables the model has
    w = W.small_config(seed=62, orders=2, fibers=2, slices=2, n_lambda=40000, n_slit=2, width=400, height=160)
    narrow = W.Workload(w.name, w.model.copy(), w.spectra, w.out_dtype, w.precision)
    for s in narrow.model.slices:
        s.sigma_x, s.sigma_y = 0.5 * s.sigma_x, 0.5 * s.sigma_y
    first = renderer.load_model(narrow.model)  # below 1 px: no polynomials
    sids = renderer.load_spectra(w)
    renderer.render(first, sids, "mixed", "f32")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    hold = torch.empty(free - (400 << 20), dtype=torch.uint8, device="cuda:0")
    second = 0
    try:
        second = renderer.load_model(w.model)
        _check(renderer, second, sids, w, "render_mixed")
        cx, cy, sx, sy = renderer.params(first)
        renderer.update(first, cx, cy, 2.0 * sx, 2.0 * sy)
        _check(renderer, first, sids, w, "render_mixed")
        del hold
        torch.cuda.empty_cache()
        renderer.update(first, cx, cy, 2.0 * sx, 2.0 * sy)
        _check(renderer, first, sids, w, "render_poly")
    finally:
        for mid in (first, second):
            if mid:
                renderer.unload_model(mid)
