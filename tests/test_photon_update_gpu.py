"""Photons of an updated model: the renderer's FP32 copy of the coefficients follows an update, so
the counts are the oracle's for the updated model, bit for bit (and the loaded model's once its
coefficients are put back)."""
import numpy as np
import pytest

import oracle
from paper_2008_05858_gb300 import workloads as W
from tests.test_photon_gpu import scaled_workload

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_counts_follow_an_update():
    from paper_2008_05858_gb300.binding import Renderer

    w = scaled_workload(W.small_config(seed=321, n_lambda=200, n_slit=9), 2e5)
    r = Renderer(0)
    try:
        mid = r.load_model(w.model)
        sids = r.load_spectra(w)
        cx, cy, sx, sy = r.params(mid)
        for scale, dy in ((1.0, 0.0), (1.25, 3.3), (1.0, 0.0)):
            ny = np.array(cy)
            o = 0
            for s in w.model.slices:
                ny[o] += dy
                ny[o + W.coeff_index(2, 0)] *= scale
                o += W.n_coeffs(s.degree)
            r.update(mid, cx, ny, sx * scale, sy * scale)
            out, total = r.render_photons(mid, sids, seed=77)
            torch.cuda.synchronize()
            ref, ref_total = oracle.render_photons(r.models[mid], w.flux_for, seed=77)
            assert total == ref_total
            for g, q in zip(out, ref):
                assert np.array_equal(g.cpu().numpy().view(np.uint32), q)
    finally:
        r.close()
