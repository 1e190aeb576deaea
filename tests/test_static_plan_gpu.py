"""Models near the fixed-scratch render's buffer: the polynomial kernel's smaller items overlap more, and
must not push a model over the 64 MiB that its edge-tail items keep to.  Box areas by hand (K = 11, 1 px a
sample along the trace, five slit points too far apart to share a run): 75 columns for an item of 64 samples,
43 for one of 32."""
import numpy as np
import pytest

import oracle
from paper_2008_05858_gb300 import workloads as W
from tests.framecompare import compare

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def straight(n_slices, slit_px, n_lambda=2048):
    """Straight traces along the frame's rows, 1 px a sample, with a five-point slit across the columns."""
    nc, slices, flux = W.n_coeffs(3), [], {}
    H = slit_px + 60
    for n in range(n_slices):
        cx, cy = np.zeros(nc), np.zeros(nc)
        cx[0], cx[W.coeff_index(1, 0)] = n_lambda / 2 + 0.13 * n, n_lambda / 2
        cy[0], cy[W.coeff_index(0, 1)] = H / 2 + 0.31 * n, (slit_px - 11) / 1.6  # the points: -0.8 .. 0.8
        slices.append(W.OrderSlice(
            detector=0, order=n + 1, fiber=0, slice=0, degree=3, K=11, n_lambda=n_lambda, n_slit=5, lambda_lo=5000.0,
            lambda_hi=5100.0, cx=cx, cy=cy, sigma_x=np.array([1.4, 0.1, 0.0]), sigma_y=np.array([1.5, 0.0, 0.0]),
            theta=0.0, slit_weights=np.array([0.5, 0.7, 1.0, 0.8, 0.6])))
        flux[n + 1] = 1000.0 + 300.0 * np.sin(0.01 * (n + 1) * np.arange(n_lambda))
    m = W.OpticalModel([(H, n_lambda)], slices, W.PSF_SEPARABLE)
    return W.Workload("straight", m, {0: W.Spectrum(0, flux)}, "f32", "mixed")


# 18 traces, 576 items of 75 x 185 px: 64 MB; one block each, as a thin grid is cut, 73 MB
# 10 traces, 320 items of 75 x 334 px: 64 MB; too large for the polynomials at two blocks, 74 MB at one
@pytest.mark.parametrize("n_slices,slit_px", [(18, 185), (10, 334)], ids=["thin_grid", "large_boxes"])
def test_model_within_the_buffer(n_slices, slit_px):
    from paper_2008_05858_gb300 import binding as B

    w = straight(n_slices, slit_px)
    r = B.Renderer(0)
    try:
        mid, sids = r.load_model(w.model), r.load_spectra(w)
        assert 60e6 < r.plan(mid)["scratch_bytes"] < B.E2E_STATIC_SCRATCH_BYTES
        ref = r.render(mid, sids, "mixed", "f32")[0]
        out = torch.full_like(ref, float("nan"))
        B.e2e_render_static(r.ctx, mid, sids, B.E2E_F32, [out.data_ptr()], [out.stride(0)])
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
        rep = compare(ref.double().cpu().numpy(), oracle.render(w.model, w.flux_for)[0])
        assert rep.ok, str(rep)
    finally:
        r.close()
