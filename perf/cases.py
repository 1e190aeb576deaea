"""What this renderer's speed is judged by: the work its users have it do, through its public
entry points, over the sizes of the repository's own configurations, tests and benchmark.

A case's "kind" is the call it makes:

  render     Renderer.render of a separable-PSF model (mixed precision to FP32 frames, or the
             plain FP64 renderer to FP64 frames)
  exposure   spectra uploaded, frame rendered into page-locked host memory, spectra unloaded
  elliptical Renderer.render of rotated Gaussian PSFs
  table      Renderer.render of tabulated PSF maps
  gradient   Renderer.adjoint for a given dL/dI
  fit        autograd.render and backward: coefficients in, frames and gradient out
  noise      Renderer.add_noise, electrons in, ADU out
  photons    Renderer.render_photons
  serve      a burst of small and medium jobs through the Server's request loop

Geometry, spectra, PSF maps and detector frames are made here from the seed alone.
"""
import math

import numpy as np
import torch

from paper_2008_05858_gb300 import autograd
from paper_2008_05858_gb300 import workloads as W
from paper_2008_05858_gb300.binding import Renderer, Server, e2e_unload_spectrum

DEV = "cuda:0"


def _case(name, kind, size, orders, fibers, slices, n_lambda, n_slit, degree, K, sigma_lo=1.2, sigma_hi=2.0, **more):
    c = dict(kind=kind, height=size[0], width=size[1], orders=orders, fibers=fibers, slices=slices,
             n_lambda=n_lambda, n_slit=n_slit, degree=degree, K=K, sigma_lo=sigma_lo, sigma_hi=sigma_hi)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one order on a 1024 x 256 tile: the serving mix's small job, where latency counts
        _case("tile_1024", "render", (256, 1024), 1, 2, 2, 2000, 16, 5, 11, precision="mixed"),
        # the plain method: one fiber of one order in FP64 (also the check on the mixed renders)
        _case("tile_fp64", "render", (256, 1024), 1, 1, 1, 2000, 16, 3, 7, 1.5, 1.5, precision="fp64"),
        # ten orders on 4096^2: the serving mix's medium job
        _case("frame_4096", "render", (4096, 4096), 10, 2, 2, 4000, 32, 5, 11, precision="mixed"),
        # a full 9216^2 detector, 85 orders x 2 fibers x 2 slices: the headline frame
        _case("frame_9216", "render", (9216, 9216), 85, 2, 2, 6000, 64, 5, 11, precision="mixed"),
        # the same frame as a streaming caller has it: new spectra in, the frame in host memory
        _case("exposure_9216", "exposure", (9216, 9216), 85, 2, 2, 6000, 64, 5, 11),
        # rotated 13 x 13 PSFs of the multi-detector instrument: three of its orders on one detector
        _case("elliptical_3", "elliptical", (9216, 9216), 3, 4, 2, 8000, 128, 5, 13, theta=10.0),
        # PSF maps from an optical design (5 field points, 10 samples per pixel)
        _case("table_4096", "table", (4096, 4096), 10, 2, 2, 4000, 32, 5, 11, fields=5, oversample=10, coma=0.1),
        # calibration fitting on a 2048^2 tile: the gradient alone, for a caller with its own loss
        _case("gradient_2048", "gradient", (2048, 2048), 10, 1, 1, 4000, 32, 4, 9),
        # ... and one iteration through torch.autograd: new coefficients, render, gradient
        _case("fit_2048", "fit", (2048, 2048), 10, 1, 1, 4000, 32, 4, 9),
        # photon, dark and read-out noise, pixel response, cross-talk and ADU of a full frame
        _case("noise_9216", "noise", (9216, 9216), 85, 2, 2, 6000, 4, 1, 11),
        # photon by photon, 1e8 of them: short exposures, where it rivals the stamp method
        _case("photons_1e8", "photons", (9216, 9216), 85, 2, 2, 6000, 64, 5, 11, photons=1e8),
        # requests that arrive together: 8 single-order tiles and 8 ten-order frames in 8 slots
        _case("serve_burst", "serve", (4096, 4096), 10, 2, 2, 4000, 32, 5, 11, jobs=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "exposure", "elliptical", "elliptical", "table", "gradient",
                       "fit", "noise", "photons", "serve"])
    w = _log(rng, 300, 9216)
    h = max(160, min(9216, _log(rng, 0.25 * w, 1.5 * w)))
    orders = max(1, min(85, _log(rng, 1, max(2, h / 108))))
    fibers, slices = rng.choice([1, 2]), rng.choice([1, 2])
    n_lambda = max(64, min(8000, int(w * rng.uniform(0.6, 1.9))))
    n_slit = _log(rng, 8, 64)
    degree = rng.choice([3, 4, 5, 5, 6])
    K = rng.choice([7, 9, 11, 11, 13])
    lo = rng.uniform(1.0, 1.4)
    hi = lo + rng.uniform(0.2, 0.8)
    c = dict(degree=degree, K=K, sigma_lo=round(lo, 3), sigma_hi=round(hi, 3))
    if kind == "render" and rng.random() < 0.25:  # the FP64 renderer is used on small tiles
        w, h = min(w, 2048), min(h, 512)
        return _case(None, kind, (h, w), min(orders, 2), 1, slices, min(n_lambda, 2500), min(n_slit, 32),
                     precision="fp64", **c)
    if kind == "render":
        return _case(None, kind, (h, w), orders, fibers, slices, n_lambda, n_slit, precision="mixed", **c)
    if kind in ("exposure", "photons"):
        if kind == "photons":
            c["photons"] = float(_log(rng, 1e6, 3e8))
        return _case(None, kind, (h, w), orders, fibers, slices, n_lambda, n_slit, **c)
    if kind == "elliptical":
        return _case(None, kind, (h, w), min(orders, 3), fibers, slices, n_lambda, rng.randint(16, 128),
                     theta=round(rng.uniform(0.0, 12.0), 2), **c)
    if kind == "table":
        return _case(None, kind, (min(h, 4096), min(w, 4096)), min(orders, 10), fibers, slices, min(n_lambda, 4000),
                     min(n_slit, 32), fields=rng.randint(2, 5), oversample=rng.choice([4, 5, 8, 10]),
                     coma=round(rng.uniform(0.0, 0.2), 3), **c)
    if kind in ("gradient", "fit"):
        return _case(None, kind, (min(h, 2048), min(w, 2048)), min(orders, 10), fibers, 1, min(n_lambda, 4000),
                     min(n_slit, 32), **c)
    if kind == "noise":
        return _case(None, kind, (h, w), orders, fibers, slices, n_lambda, 4, 1, c["K"])
    return _case(None, kind, (min(h, 4096), min(w, 4096)), min(orders, 10), fibers, slices, min(n_lambda, 4000),
                 min(n_slit, 32), jobs=rng.randint(2, 12), **c)


# ------------------------------------------------------------------ inputs


def _idx(a, b):
    return (a + b) * (a + b + 1) // 2 + b


def _traces(case, seed, height=None, width=None, orders=None, n_lambda=None, n_slit=None):
    """The optical model's traces as plain arrays: gently curved orders across the detector,
    fibers x slices traces 16 px apart in each."""
    rng = np.random.default_rng([int(seed), 1])
    H, Wd = height or case["height"], width or case["width"]
    n_o, d = orders or case["orders"], case["degree"]
    lo, hi = case["sigma_lo"], case["sigma_hi"]
    n_tr = case["fibers"] * case["slices"]
    out = []
    for o in range(n_o):
        order = 90 + o
        theta = math.radians(rng.uniform(-1, 1) * case.get("theta", 0.0))
        lam_c = 6.0e5 / order
        half = 0.6 * lam_c / order
        for i in range(n_tr):
            nc = (d + 1) * (d + 2) // 2
            cx, cy = np.zeros(nc), np.zeros(nc)
            for t in range(2, d + 1):
                for b in range(t + 1):
                    cx[_idx(t - b, b)], cy[_idx(t - b, b)] = rng.uniform(-1, 1, 2) * 2.0 ** -t
            cx[0], cy[0] = Wd / 2.0, (o + 0.5) * H / n_o + (i - (n_tr - 1) / 2.0) * 16.0
            if d >= 1:
                cx[_idx(1, 0)], cx[_idx(0, 1)] = 0.45 * Wd, rng.uniform(-1, 1)
                cy[_idx(1, 0)], cy[_idx(0, 1)] = 0.5 * rng.uniform(-1, 1), 4.0
            if d >= 2:
                cy[_idx(2, 0)] = rng.uniform(5.0, 20.0)
            sig = []
            for _ in range(2):
                c0 = rng.uniform(0.625 * lo + 0.375 * hi, 0.375 * lo + 0.625 * hi)
                room = min(c0 - lo, hi - c0)
                c1 = rng.uniform(-0.5, 0.5) * room
                sig.append(np.array([c0, c1, rng.uniform(-0.5, 0.5) * (room - abs(c1))]))
            out.append(dict(order=order, fiber=i // case["slices"], slice=i % case["slices"], degree=d, K=case["K"],
                            n_lambda=n_lambda or case["n_lambda"], n_slit=n_slit or case["n_slit"], lo=lam_c - half,
                            hi=lam_c + half, cx=cx, cy=cy, sx=sig[0], sy=sig[1], theta=theta))
    return out


def _spectra(traces, seed):
    """{fiber: {order: photons per Angstrom}}: the even fibers carry a line-rich absorption
    spectrum, the odd ones a Fabry-Perot comb equally spaced in velocity."""
    rng = np.random.default_rng([int(seed), 2])
    flux = {}
    for s in traces:
        rows = flux.setdefault(s["fiber"], {})
        if s["order"] in rows:
            continue
        n, step = s["n_lambda"], (s["hi"] - s["lo"]) / s["n_lambda"]
        lam = s["lo"] + (np.arange(n) + 0.5) * step
        if s["fiber"] % 2:
            rows[s["order"]] = 2.0e3 / (1.0 + (20.0 / np.pi) ** 2
                                        * np.sin(np.pi * np.log(lam / 3000.0) / np.log1p(10.0 / 299792.458)) ** 2)
            continue
        m = 235
        centre, depth, sig = rng.uniform(s["lo"], s["hi"], m), rng.uniform(0.1, 0.9, m), rng.uniform(0.02, 0.1, m)
        r = int(0.6 / step) + 1
        at = np.rint((centre - s["lo"]) / step).astype(np.int64)[:, None] + np.arange(-r, r + 1)
        z = (s["lo"] + (at + 0.5) * step - centre[:, None]) / sig[:, None]
        dip = np.log1p(-depth[:, None] * np.exp(-0.5 * z * z))
        ok = (at >= 0) & (at < n)
        rows[s["order"]] = rng.uniform(1.0e3, 3.0e3) * np.exp(np.bincount(at[ok], dip[ok], n))
    return flux


def _maps(s, case):
    """PSF maps at the field points: the trace's Gaussian plus a fainter displaced one (coma)."""
    q, F = case["oversample"], case["fields"]
    M = 16 * q + 1
    x = (np.arange(M) - (M - 1) / 2.0) / q
    lt = np.linspace(-1.0, 1.0, F)
    maps = np.empty((F, M, M))
    for f in range(F):
        sx, sy = (c[0] + c[1] * lt[f] + c[2] * lt[f] ** 2 for c in (s["sx"], s["sy"]))
        gx, gy = np.exp(-0.5 * (x / sx) ** 2) / sx, np.exp(-0.5 * (x / sy) ** 2) / sy
        g2 = np.exp(-0.5 * ((x - 1.5 * sx) / (1.3 * sx)) ** 2) / (1.3 * sx)
        maps[f] = np.outer(gy, (1 - case["coma"]) * gx + case["coma"] * g2) / (2 * np.pi)
    return lt, maps


def _model(case, traces, height=None, width=None):
    psf = {"elliptical": W.PSF_ELLIPTICAL, "table": W.PSF_TABLE}.get(case["kind"], W.PSF_SEPARABLE)
    out = []
    for s in traces:
        pm = W.PsfMap(*_maps(s, case), float(case["oversample"])) if case["kind"] == "table" else None
        out.append(W.OrderSlice(
            detector=0, order=s["order"], fiber=s["fiber"], slice=s["slice"], degree=s["degree"], K=s["K"],
            n_lambda=s["n_lambda"], n_slit=s["n_slit"], lambda_lo=s["lo"], lambda_hi=s["hi"], cx=s["cx"], cy=s["cy"],
            sigma_x=s["sx"], sigma_y=s["sy"], theta=s["theta"], slit_weights=np.full(s["n_slit"], 1.0 / s["n_slit"]),
            psf_map=pm))
    return W.OpticalModel([(height or case["height"], width or case["width"])], out, psf)


def _electrons(case, seed):
    """Expected electrons of an exposure: bright, curved traces over a faint background."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) % (1 << 62))
    H, Wd, n = case["height"], case["width"], case["orders"]
    y = torch.arange(H, device=DEV, dtype=torch.float32)[:, None]
    x = torch.linspace(-1, 1, Wd, device=DEV)[None, :]
    band = H / n
    frame = torch.empty((H, Wd), device=DEV)
    rows = max(1, (1 << 26) // Wd)
    tilt = 10.0 * torch.rand(1, device=DEV, generator=g)
    amp = 4.0e4 * torch.rand((n + 1, Wd), device=DEV, generator=g) ** 2
    for r in range(0, H, rows):
        v = y[r:r + rows] + tilt * x * x
        o = torch.clamp((v / band).floor().long(), 0, n)
        off = (v - (o + 0.5) * band) / 4.0
        frame[r:r + rows] = 0.05 + torch.gather(amp, 0, o.expand(-1, Wd)) * torch.exp(-0.5 * off * off)
    return frame


def _dldi(case, seed):
    """dL/dI as a least-squares fit has it: the residuals' noise about zero."""
    g = torch.Generator(device=DEV).manual_seed((int(seed) + 77) % (1 << 62))
    return torch.randn((case["height"], case["width"]), device=DEV, generator=g) * 3.0


def _pinned(shape):
    """A page-locked host frame."""
    return torch.empty(shape, dtype=torch.float32, pin_memory=True)


class State(dict):
    """What the program keeps; its context is closed with it."""

    def __del__(self):
        if "server" in self:
            self["server"].stop()
        if "r" in self:
            self["r"].close()


def prepare(case, seed):
    kind = case["kind"]
    s = State(kind=kind, r=Renderer(0))
    r = s["r"]
    if kind == "serve":
        s["jobs"] = []
        kinds = [dict(height=256, width=1024, orders=1, n_lambda=2000, n_slit=16), {}]
        for i, over in enumerate(kinds):
            tr = _traces(case, seed + i, **over)
            mid = r.load_model(_model(case, tr, over.get("height"), over.get("width")))
            sids = [r.load_spectrum(W.Spectrum(f, o)) for f, o in sorted(_spectra(tr, seed + i).items())]
            s["jobs"] += [(mid, sids, r.empty_frames(mid)) for _ in range(case["jobs"])]
        s["jobs"] = s["jobs"][::2] + s["jobs"][1::2]
        s["server"] = Server(r, max_inflight=8)
        return s
    traces = _traces(case, seed)
    s["mid"] = r.load_model(_model(case, traces))
    if kind == "noise":
        s["frames"] = [_electrons(case, seed)]
        s["out"] = [torch.empty((case["height"], case["width"]), dtype=torch.uint16, device=DEV)]
        s["seed"] = int(seed) % (1 << 31)
        return s
    spectra = _spectra(traces, seed)
    if kind == "photons":  # spectra scaled to the expected number of photons
        dl = {t["order"]: (t["hi"] - t["lo"]) / t["n_lambda"] for t in traces}
        tot = sum(float(spectra[t["fiber"]][t["order"]].sum()) * dl[t["order"]] for t in traces)
        spectra = {f: {o: v * (case["photons"] / tot) for o, v in rows.items()} for f, rows in spectra.items()}
        s["seed"] = int(seed) % (1 << 31)
        s["out"] = [torch.empty((case["height"], case["width"]), dtype=torch.int32, device=DEV)]
    if kind == "exposure":
        s["spectra"] = [W.Spectrum(f, o) for f, o in sorted(spectra.items())]
        s["out"] = [_pinned((case["height"], case["width"]))]
        return s
    s["sids"] = [r.load_spectrum(W.Spectrum(f, o)) for f, o in sorted(spectra.items())]
    if kind == "render":
        s["precision"] = case["precision"]
        s["dtype"] = "f64" if case["precision"] == "fp64" else "f32"
        s["out"] = r.empty_frames(s["mid"], s["dtype"])
    elif kind in ("elliptical", "table"):
        s["precision"], s["dtype"] = "mixed", "f32"
        s["out"] = r.empty_frames(s["mid"])
    elif kind in ("gradient", "fit"):
        s["dldi"] = [_dldi(case, seed)]
        if kind == "fit":
            s["params"] = torch.tensor(autograd.pack(r.params(s["mid"])), dtype=torch.float64, requires_grad=True)
    return s


# ------------------------------------------------------------------ the calls


def run(s):
    r, kind = s["r"], s["kind"]
    if kind == "exposure":
        sids = [r.load_spectrum(sp) for sp in s["spectra"]]
        r.render_host(s["mid"], sids, out=s["out"])
        for i in sids:
            e2e_unload_spectrum(r.ctx, i)
        return s["out"]
    if kind == "gradient":
        return list(r.adjoint(s["mid"], s["sids"], s["dldi"]))
    if kind == "fit":
        s["params"].grad = None
        frames = autograd.render(s["params"], r, s["mid"], s["sids"])
        torch.autograd.backward(frames, s["dldi"])
        return {"frames": [f.detach() for f in frames], "gradient": s["params"].grad}
    if kind == "noise":
        adu = r.add_noise(s["mid"], s["frames"], "u16", out=s["out"], seed=s["seed"], pattern_seed=17, dark_e=2.5,
                          prnu=0.01, ron_e=3.2, xtalk=2e-4, gain=1.1, bias=300.0)
        return [f.view(torch.int16) for f in adu]  # the same bits: torch cannot index unsigned 16-bit tensors
    if kind == "photons":
        frames, total = r.render_photons(s["mid"], s["sids"], s["seed"], out=s["out"])
        return {"frames": frames, "total": total}
    if kind == "serve":
        srv = s["server"]
        ids = [srv.submit(mid, sids, out=out) for mid, sids, out in s["jobs"]]
        for i in ids:
            srv.wait(i)
            srv.forget(i)
        return [out for _, _, out in s["jobs"]]
    return r.render(s["mid"], s["sids"], s["precision"], s["dtype"], out=s["out"])


def work(case):
    """Spectra (FP64) in and frames out once; per stamp the K x K window's multiply-adds."""
    px = case["height"] * case["width"]
    stamps = case["orders"] * case["fibers"] * case["slices"] * case["n_lambda"] * case["n_slit"]
    spec = 8 * case["orders"] * case["fibers"] * case["n_lambda"]
    k2 = case["K"] ** 2
    kind = case["kind"]
    if kind == "noise":
        return {"bytes": 6 * px, "flops": 0}
    if kind == "photons":
        return {"bytes": 4 * px + spec, "flops": 2 * case["photons"] * (case["degree"] + 1) * (case["degree"] + 2)}
    if kind == "gradient":  # each window pixel enters the column and the row sums
        return {"bytes": 4 * px + spec, "flops": 4 * k2 * stamps}
    if kind == "fit":
        return {"bytes": 8 * px + spec, "flops": 6 * k2 * stamps}
    if kind == "serve":
        small = case["fibers"] * case["slices"] * 2000 * 16
        return {"bytes": case["jobs"] * (4 * (px + 256 * 1024) + spec), "flops": case["jobs"] * 2 * k2 * (stamps + small)}
    size = 8 if case.get("precision") == "fp64" else 4
    return {"bytes": size * px + spec, "flops": 2 * k2 * stamps}


# ------------------------------------------------------------------ the same in 64 bits

_R2 = math.sqrt(0.5)


def _between(a, b):
    """P(a < Z < b) of a standard normal, without cancellation against 1."""
    ea, eb = torch.special.erfc(a.abs() * _R2), torch.special.erfc(b.abs() * _R2)
    return torch.where(a >= 0, 0.5 * (ea - eb), torch.where(b <= 0, 0.5 * (eb - ea), 1.0 - 0.5 * (ea + eb)))


def _edges(v, i0, K, sig):
    """Window edges (n, K + 1) in units of sigma about v."""
    e = i0[:, None] + torch.arange(K + 1, device=DEV) - 0.5
    return (e - v[:, None]) / sig[:, None]


def _stamps(case, traces, flux, per_stamp):
    """Blocks of stamps (trace, sample and slit indices, weights, centres, window origins)."""
    for s in traces:
        n_l, n_s, d, K = s["n_lambda"], s["n_slit"], s["degree"], s["K"]
        f = torch.tensor(flux[s["fiber"]][s["order"]], device=DEV, dtype=torch.float64)
        step = max(1, int(1.0e8 / per_stamp / n_s))
        ss = (2 * torch.arange(n_s, device=DEV, dtype=torch.float64) + 1 - n_s) / n_s
        for j0 in range(0, n_l, step):
            j = torch.arange(j0, min(n_l, j0 + step), device=DEV)
            lt = (2 * j.double() + 1 - n_l) / n_l
            x, y = (sum(float(c[_idx(a, b)]) * lt[:, None] ** a * ss[None, :] ** b
                        for a in range(d + 1) for b in range(d + 1 - a)) for c in (s["cx"], s["cy"]))
            w = (f[j] * ((s["hi"] - s["lo"]) / n_l) / n_s)[:, None].expand_as(x)
            lt, sv = lt[:, None].expand_as(x).reshape(-1), ss[None, :].expand_as(x).reshape(-1)
            x, y, w = x.reshape(-1), y.reshape(-1), w.reshape(-1)
            i0, r0 = (torch.floor(v + 0.5).long() - K // 2 for v in (x, y))
            sx, sy = (c[0] + c[1] * lt + c[2] * lt * lt for c in (s["sx"], s["sy"]))
            yield s, lt, sv, x, y, w, i0, r0, sx, sy


def _add(frame, val, i0, r0, K):
    H, Wd = frame.shape
    k = torch.arange(K, device=DEV)
    r, c = r0[:, None, None] + k[:, None], i0[:, None, None] + k
    ok = (r >= 0) & (r < H) & (c >= 0) & (c < Wd)
    frame.view(-1).index_add_(0, torch.where(ok, r * Wd + c, 0).view(-1), torch.where(ok, val, 0.0).view(-1))


def _exact_frame(case, seed, traces=None, shape=None):
    traces = traces or _traces(case, seed)
    flux, K = _spectra(traces, seed), case["K"]
    frame = torch.zeros(shape or (case["height"], case["width"]), device=DEV, dtype=torch.float64)
    for s, lt, _, x, y, w, i0, r0, sx, sy in _stamps(case, traces, flux, 4 * K * K):
        ex, ey = _edges(x, i0, K, sx), _edges(y, r0, K, sy)
        ax, ay = _between(ex[:, :-1], ex[:, 1:]) * w[:, None], _between(ey[:, :-1], ey[:, 1:])
        _add(frame, ay[:, :, None] * ax[:, None, :], i0, r0, K)
    return frame


def _exact_elliptical(case, seed):
    """Gauss-Legendre over each pixel column of the x-marginal times the conditional interval in y."""
    traces = _traces(case, seed)
    flux, K = _spectra(traces, seed), case["K"]
    frame = torch.zeros((case["height"], case["width"]), device=DEV, dtype=torch.float64)
    t, gw = (torch.tensor(v * 0.5, device=DEV) for v in np.polynomial.legendre.leggauss(8))
    for s, lt, _, x, y, w, i0, r0, sa, sb in _stamps(case, traces, flux, 40 * K * K):
        c, n = math.cos(s["theta"]), math.sin(s["theta"])
        vx, vy, cxy = (sa * c) ** 2 + (sb * n) ** 2, (sa * n) ** 2 + (sb * c) ** 2, (sa ** 2 - sb ** 2) * n * c
        beta = cxy / vx
        sc = torch.sqrt(vy - beta * cxy)
        val = torch.zeros((len(x), K, K), device=DEV, dtype=torch.float64)
        for q in range(len(t)):
            u = i0[:, None] + torch.arange(K, device=DEV) + t[q] - x[:, None]
            px = gw[q] * torch.exp(-0.5 * u * u / vx[:, None]) / torch.sqrt(2 * math.pi * vx)[:, None]
            mid = y[:, None] + beta[:, None] * u
            e = (r0[:, None, None] + torch.arange(K + 1, device=DEV)[:, None] - 0.5 - mid[:, None, :]) / sc[:, None, None]
            val += px[:, None, :] * _between(e[:, :-1], e[:, 1:])
        _add(frame, val * w[:, None, None], i0, r0, K)
    return frame


def _tent_cdf(t):
    t = t.clamp(-1.0, 1.0)
    return torch.where(t <= 0, 0.5 * (1 + t) ** 2, 1 - 0.5 * (1 - t) ** 2)


def _exact_table(case, seed):
    """The bilinear maps integrated over each pixel about the exact centre, blended in lt."""
    traces = _traces(case, seed)
    flux, K = _spectra(traces, seed), case["K"]
    frame = torch.zeros((case["height"], case["width"]), device=DEV, dtype=torch.float64)
    q, F, held = case["oversample"], case["fields"], {}
    for s, lt, _, x, y, w, i0, r0, _, _ in _stamps(case, traces, flux, 24 * K * (16 * q + 1)):
        if held.get("of") is not s:
            maps = torch.tensor(_maps(s, case)[1], device=DEV)
            held = {"of": s, "maps": maps / maps.sum((1, 2), keepdim=True) * q * q}
        M = 16 * q + 1
        at = (torch.arange(M, device=DEV, dtype=torch.float64) - (M - 1) / 2.0) / q
        px, py = (torch.diff(_tent_cdf(q * ((o[:, None] + torch.arange(K + 1, device=DEV) - 0.5 - v[:, None])[:, :, None]
                                            - at)), dim=1) / q for o, v in ((i0, x), (r0, y)))
        pos = (lt + 1.0) * (F - 1) / 2.0
        val = 0.0
        for f in range(F):
            blend = (1.0 - (pos - f).abs()).clamp(min=0.0)
            if float(blend.max()) > 0.0:
                rows = torch.matmul(py.view(-1, M), held["maps"][f]).view(-1, K, M)
                val = val + torch.matmul(rows, px.transpose(1, 2)) * blend[:, None, None]
        _add(frame, val * w[:, None, None], i0, r0, K)
    return frame


def _exact_gradient(case, seed):
    traces = _traces(case, seed)
    flux, K, R = _spectra(traces, seed), case["K"], _dldi(case, seed).double()
    H, Wd = R.shape
    g = {k: [torch.zeros(len(t[k]), device=DEV, dtype=torch.float64) for t in traces] for k in ("cx", "cy", "sx", "sy")}
    at = {id(t): i for i, t in enumerate(traces)}
    k = torch.arange(K, device=DEV)
    for s, lt, sv, x, y, w, i0, r0, sx, sy in _stamps(case, traces, flux, 6 * K * K):
        r, c = r0[:, None, None] + k[:, None], i0[:, None, None] + k
        ok = (r >= 0) & (r < H) & (c >= 0) & (c < Wd)
        patch = torch.where(ok, R.view(-1)[torch.where(ok, r * Wd + c, 0)], 0.0)
        e = [_edges(x, i0, K, sx), _edges(y, r0, K, sy)]
        A = [_between(u[:, :-1], u[:, 1:]) for u in e]
        phi = [torch.exp(-0.5 * u * u) / math.sqrt(2 * math.pi) for u in e]
        dA = [-torch.diff(p, dim=1) / v[:, None] for p, v in zip(phi, (sx, sy))]
        sA = [-torch.diff(p * u, dim=1) / v[:, None] for p, u, v in zip(phi, e, (sx, sy))]
        S = [torch.einsum("nrc,nr->nc", patch, A[1]), torch.einsum("nrc,nc->nr", patch, A[0])]
        for z, name, wide in ((0, "cx", "sx"), (1, "cy", "sy")):
            gc_, gs = (w * (D[z] * S[z]).sum(1) for D in (dA, sA))
            for a in range(s["degree"] + 1):
                for b in range(s["degree"] + 1 - a):
                    g[name][at[id(s)]][_idx(a, b)] += (gc_ * lt ** a * sv ** b).sum()
            for a in range(3):
                g[wide][at[id(s)]][a] += (gs * lt ** a).sum()
    return [torch.cat(g[name]) for name in ("cx", "cy", "sx", "sy")]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("render", "exposure"):
        return [_exact_frame(case, seed)]
    if kind == "elliptical":
        return [_exact_elliptical(case, seed)]
    if kind == "table":
        return [_exact_table(case, seed)]
    if kind == "gradient":
        return _exact_gradient(case, seed)
    if kind == "fit":
        return {"frames": [_exact_frame(case, seed)], "gradient": torch.cat(_exact_gradient(case, seed))}
    if kind == "serve":
        over = dict(height=256, width=1024, orders=1, n_lambda=2000, n_slit=16)
        small = _exact_frame(case, seed, _traces(case, seed, **over), (256, 1024))
        medium = _exact_frame(case, seed + 1, _traces(case, seed + 1))
        jobs = [[small]] * case["jobs"] + [[medium]] * case["jobs"]
        return jobs[::2] + jobs[1::2]
    return None  # noise and photon counts are whole numbers
