"""The separable render on polynomial pixel integrals (models whose widths stay >= 1 px) against
the oracle, where it can go wrong: every window size, runs cut short by the slit, widths on
either side of the table's limit, strongly curved and falling slits (exact mapping, tile origins),
samples beyond a multiple of a warp's eight, frames narrower than a window."""
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


def _slit(c, slope, curve):
    """The slices' slits re-pointed: s^1 coefficient of y, s^2 coefficient of x and y."""
    for s in c.slices:
        s.cy[W.coeff_index(0, 1)] = slope
        s.cx[W.coeff_index(0, 2)] = curve
        s.cy[W.coeff_index(0, 2)] = curve


CASES = [(f"K{K}", dict(seed=300 + K, K=K, n_lambda=97, n_slit=17), None) for K in (3, 5, 7, 9, 11, 13, 15)]
CASES += [(f"slit{n}", dict(seed=320 + n, n_lambda=41, n_slit=n), None) for n in (1, 2, 3, 8, 15, 31, 64, 129)]
CASES += [
    ("width_1.0", dict(seed=341, sigma_range=(1.0, 1.0 + 1e-9)), None),
    ("width_below_1", dict(seed=342, sigma_range=(0.96, 0.999)), None),
    ("width_wide", dict(seed=343, sigma_range=(2.0, 6.0), K=15), None),
    ("samples_1", dict(seed=344, n_lambda=1), None),
    ("samples_9", dict(seed=345, n_lambda=9), None),
    ("degree_0", dict(seed=346, degree=0, K=7), None),
    ("degree_1", dict(seed=347, degree=1, K=9), None),
    ("degree_8", dict(seed=348, degree=8), None),
    ("falling_slit", dict(seed=349, n_slit=32), lambda m: _slit(m, -5.0, 0.0)),
    ("curved_slit", dict(seed=350, n_slit=32), lambda m: _slit(m, 4.0, 2.5)),
    ("steep_slit", dict(seed=351, n_slit=16, width=200, height=200), lambda m: _slit(m, 70.0, 0.5)),
    ("narrow_frame", dict(seed=352, width=8, height=40, n_lambda=40), None),
]


@pytest.mark.parametrize("kw,change", [c[1:] for c in CASES], ids=[c[0] for c in CASES])
def test_matches_oracle(kw, change):
    w = W.small_config(**kw)
    if change is not None:
        change(w.model)
    got, checked = _frames(w, 0), _frames(w, 1)
    ref = oracle.render_workload(w)
    for g, c, o in zip(got, checked, ref):
        rep = compare(g, o)
        assert rep.ok, rep
        assert np.array_equal(g, c)  # the checking build deposits the same
