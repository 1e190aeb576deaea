"""The tabulated-PSF render whose stamps are sorted by phase cell, against the oracle, at the edges
of the sort: more cells than stamps and one cell, slices of unlike cell counts, field nodes that
change within an item (a cell's stamps then read unlike tables), one node, one sample, one slit
point, and a work item whose box leaves no room to sort.  The separable renderer's tolerance."""
import numpy as np
import pytest

import oracle
from paper_2008_05858_gb300 import workloads as W
from tests.framecompare import compare

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [
    ("cells_1089", dict(seed=731, n_lambda=64), dict(oversample=32.0, even_size=True)),
    ("cells_1", dict(seed=732, n_lambda=90), dict(oversample=1.0)),
    ("unlike_slices", dict(seed=733, n_lambda=90), None),
    ("fields_25", dict(seed=734, n_lambda=120), dict(oversample=4.0, n_field=25)),
    ("field_1", dict(seed=735, n_lambda=70), dict(oversample=4.0, n_field=1)),
    ("sample_1", dict(seed=736, n_lambda=1), dict(oversample=3.0)),
    ("slit_1", dict(seed=737, n_lambda=33, n_slit=1), dict(oversample=3.0)),
    ("slit_17", dict(seed=738, n_lambda=33, n_slit=17), dict(oversample=3.0)),
    ("window_1", dict(seed=739, K=1, n_lambda=70), dict(oversample=4.0)),
    ("window_15", dict(seed=740, K=15, n_lambda=70), dict(oversample=4.0)),
    # one item spans the frame: 26,880 box pixels leave less than the sort's 18 KB
    ("no_room", dict(seed=741, width=120, height=224, orders=1, fibers=1, slices=1, n_lambda=32, n_slit=16),
     dict(oversample=5.0)),
]


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


@pytest.mark.parametrize("name,kw,maps", CASES, ids=[c[0] for c in CASES])
def test_matches_oracle(name, kw, maps):
    w = W.small_config(**kw)
    m = W.with_psf_maps(w.model, coma=0.2, half_px=6.0, **(maps or {}))
    if maps is None:  # another oversampling per slice
        for i, s in enumerate(m.slices):
            s.psf_map = W.psf_maps(s, oversample=float(1 + 3 * i), half_px=6.0, even_size=i % 2 == 1)
    if name == "no_room":
        for s in m.slices:
            s.cy[W.coeff_index(0, 1)] = 130.0
    w = W.Workload(w.name, m, w.spectra, "f32", "mixed")
    got, checked = _frames(w, 0), _frames(w, 1)
    for g, c, o in zip(got, checked, oracle.render_workload(w)):
        rep = compare(g, o)
        assert rep.ok, str(rep)
        assert np.array_equal(g, c)
