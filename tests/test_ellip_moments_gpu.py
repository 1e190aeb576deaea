"""The elliptical render on run moments (widths >= 1 px that vary slowly from sample to sample)
against the oracle, where it can go wrong: every window size, slits cut into parts, more runs in a
sample than are turned into pixels at once, runs of one stamp, widths between the nodes, samples
short of a warp's or an interval's, traces over the frame's edge."""
import numpy as np
import pytest

import oracle
from paper_2008_05858_gb300 import workloads as W
from tests.framecompare import compare

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _frames(w, checks):
    from paper_2008_05858_gb300.binding import Renderer

    r = Renderer(0, debug_checks=checks)
    try:
        mid = r.load_model(w.model)
        out = r.render(mid, r.load_spectra(w), "mixed", "f32")
        torch.cuda.synchronize()
        return [t.double().cpu().numpy() for t in out]
    finally:
        r.close()


def _model(seed, sig=(1.3, 1.9), theta_deg=8.0, slope=None, tilt=None, vary=None, **kw):
    kw = {**dict(orders=1, fibers=1, slices=2, n_lambda=64, n_slit=16, width=200, height=100), **kw}
    w = W.small_config(seed=seed, psf=W.PSF_ELLIPTICAL, **kw)
    for q, s in enumerate(w.model.slices):
        s.theta = np.deg2rad(theta_deg * (1 if q % 2 == 0 else -1))
        s.sigma_x = np.array([sig[0], 0.0, 0.0]) if vary is None else np.array([sig[0], vary, -0.5 * vary])
        s.sigma_y = np.array([sig[1], 0.0, 0.0]) if vary is None else np.array([sig[1], -vary, 0.5 * vary])
        if slope is not None:
            s.cy[W.coeff_index(0, 1)] = slope
        if tilt is not None:
            s.cx[W.coeff_index(0, 1)] = tilt
    return w


CASES = [(f"K{K}", dict(seed=400 + K, K=K)) for K in (3, 5, 7, 9, 11, 13, 15)]
CASES += [(f"slit{n}", dict(seed=420 + n, K=13, n_lambda=33, n_slit=n)) for n in (1, 2, 15, 17, 31, 33, 128, 129, 200)]
CASES += [
    ("many_runs", dict(seed=441, K=11, n_slit=60, n_lambda=20, slope=25.0, height=140)),
    ("falling_slit", dict(seed=442, K=9, n_slit=40, slope=-6.0, tilt=-3.0)),
    ("samples_1", dict(seed=443, n_lambda=1)),
    ("samples_95", dict(seed=444, n_lambda=95)),
    ("narrow", dict(seed=445, sig=(1.0, 1.0), theta_deg=0.0, K=7)),
    ("correlated", dict(seed=446, sig=(2.0, 1.2), theta_deg=19.0, K=13)),
    ("varying", dict(seed=447, slices=1, n_lambda=3000, n_slit=3, width=1200, K=11, vary=0.08)),
    ("varying_fast", dict(seed=448, slices=1, n_lambda=300, n_slit=5, K=9, vary=0.2, theta_deg=3.0)),  # stamp by stamp
    ("narrow_frame", dict(seed=449, width=9, height=30, n_lambda=40)),
]


@pytest.mark.parametrize("kw", [c[1] for c in CASES], ids=[c[0] for c in CASES])
def test_matches_oracle(kw):
    w = _model(**kw)
    got, checked = _frames(w, 0), _frames(w, 1)
    ref = oracle.render_workload(w)
    for g, c, o in zip(got, checked, ref):
        rep = compare(g, o)
        assert rep.ok, rep
        assert np.array_equal(g, c)  # the checked render deposits the same
