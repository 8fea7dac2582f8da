"""The work whose speed counts, as a user's program asks for it through the package's entry points.

Each case names a `kind` of call and its sizes:

  event       one event over a slice of a resident bank: submit, wait, evidence, marginals, release
  batch       several events over one bank as one launch sequence
  rb          relative-binning weights from full-resolution data, then an event that uses them
  precessing  one event over a polarisation-resolved bank
  presel      the single-detector pre-selection of a mode bank
  presel_pol  the same of a polarisation-resolved bank with relative-binning weights
  samples     posterior draws from a finished, stored event

Inputs are synthetic, with the distributions that the path meets: leading-order
chirps of 5 to 30 solar masses on log-spaced bins, prior-drawn (or, with
relative binning, concentrated) extrinsic samples, an injected bank member plus
Gaussian noise.  `exact` evaluates the same quantities in 64 bits with plain
torch.
"""
import math

import numpy as np
import torch

import paper_2507_16022_gb300 as dp

CUT = 20.0        # the paper's coherent-ML and pre-selection window
N_FINE = 131072   # points of the full-resolution grid of relative binning
GM_SUN_S = 4.925491025543576e-06
C_LIGHT, R_EARTH = 299792458.0, 6.371e6
MODES = {1: ((2, 2),), 2: ((2, 2), (3, 3)), 3: ((2, 2), (3, 3), (4, 4)), 4: ((2, 1), (2, 2), (3, 3), (4, 4))}
SITES = ((46.455, -119.408, 324.0, 234.0), (30.563, -90.774, 252.3, 162.3), (43.631, 10.504, 70.6, 340.6))
PSD_SCALE = (1.0, 1.3, 1.7)


def listed():
    return [
        # a first look at a small bank: every pair kept and read back, the binding's default precision;
        # latency and launches count
        dict(name="small_all_pairs", kind="event", bank=1024, rows=1024, ext=256, det=2, modes=3, bins=256, phases=32,
             snr=15.0, precision="bf16x3", cut=0.0, store=True, block=0, host=True),
        # an ordinary request of the serving loop: a ragged slice of a resident bank, inputs in host memory
        dict(name="served_slice", kind="event", bank=50021, rows=40037, ext=2743, det=2, modes=4, bins=256, phases=32,
             snr=30.0, precision="mixed", cut=CUT, store=False, block=0, host=True),
        # one event at production size in the served precision (the benchmark's own workload)
        dict(name="production", kind="event", bank=65536, rows=65536, ext=4096, det=3, modes=4, bins=512, phases=32,
             snr=15.0, precision="mixed", cut=CUT, store=False, block=0, host=False),
        # the plain FP32 path that other precisions are checked against, best ln L of every pair read back
        dict(name="plain_fp32", kind="event", bank=8192, rows=8192, ext=1024, det=3, modes=4, bins=512, phases=32,
             snr=15.0, precision="fp32", cut=CUT, store=True, block=0, host=False),
        # no cut, importance weights, split precision: every phase of every pair marginalised, odd sizes
        dict(name="uncut_split", kind="event", bank=12289, rows=12289, ext=771, det=3, modes=4, bins=384, phases=32,
             snr=15.0, precision="fp16x3", cut=0.0, store=True, block=0, host=False),
        # a bank larger than one pass, streamed in blocks, loud signal
        dict(name="streamed_bank", kind="event", bank=262144, rows=262144, ext=2048, det=3, modes=4, bins=384, phases=32,
             snr=30.0, precision="mixed", cut=CUT, store=False, block=65536, host=False),
        # a batch over a shared bank: extrinsic counts, detectors and loudness differ from event to event
        dict(name="batch_of_12", kind="batch", bank=65536, events=12, ext=2304, modes=4, bins=512, phases=32,
             precision="mixed", cut=CUT),
        # the paper's binning: weights on 378 nodes, bank and samples concentrated on the signal
        dict(name="relative_binning", kind="rb", rows=32768, ext=2048, det=3, modes=4, bins=378, phases=32, snr=15.0,
             precision="mixed", cut=CUT),
        # the general waveform: both polarisations of every mode held by the bank
        dict(name="precessing", kind="precessing", rows=16384, ext=4096, det=3, modes=4, bins=512, phases=32, snr=15.0,
             precision="mixed", cut=CUT),
        # the stage before the coherent evaluation: a whole bank against a time grid
        dict(name="preselect", kind="presel", rows=65536, times=128, det=3, modes=4, bins=512, phases=32, snr=15.0,
             precision="fp16x3"),
        # the paper's own pre-selection: polarisation-resolved bank and relative binning, which run in FP32
        dict(name="preselect_precessing", kind="presel_pol", rows=16384, times=128, det=3, modes=4, bins=378, phases=32,
             snr=15.0, precision="fp32"),
        # draws for one event's posterior, a few hundred at a time
        dict(name="posterior_draws", kind="samples", rows=16384, ext=2048, det=3, modes=4, bins=512, phases=32, snr=15.0,
             draws=512),
    ]


def draw(rng):
    def size(lo, hi):  # spread over the logarithm, odd sizes as often as even ones
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["event", "event", "event", "uncut", "fp32", "batch", "rb", "precessing", "presel", "presel_pol",
                       "samples"])
    modes, det = rng.choice([2, 3, 4, 4]), rng.choice([2, 3])
    bins = size(192, 512)
    phases = rng.choice([16, 32, 32, 64])
    snr = round(rng.uniform(8.0, 40.0), 2)
    if kind == "event":
        rows = size(4096, 262144)
        ext = size(256, min(8192, 2 ** 28 // rows))
        block = 65536 if rows > 131072 else 0
        return dict(kind="event", bank=rows + rng.randrange(0, 2048), rows=rows, ext=ext, det=det, modes=modes, bins=bins,
                    phases=phases, snr=snr, precision="mixed", cut=CUT, store=False, block=block,
                    host=rng.random() < 0.5)
    if kind in ("uncut", "fp32"):
        rows = size(512, 8192)
        ext = size(64, min(1024, 2 ** 23 // rows))
        return dict(kind="event", bank=rows, rows=rows, ext=ext, det=det, modes=modes, bins=min(bins, 384 if kind == "uncut" else 512),
                    phases=min(phases, 32), snr=snr,
                    precision="fp32" if kind == "fp32" else rng.choice(["bf16x3", "fp16x3"]),
                    cut=CUT if kind == "fp32" else 0.0, store=True, block=0, host=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind="batch", bank=size(8192, 65536), events=rng.randrange(3, 13), ext=size(384, 2304), modes=modes,
                    bins=bins, phases=phases, precision="mixed", cut=CUT)
    if kind == "rb":
        return dict(kind="rb", rows=size(2048, 32768), ext=size(256, 2048), det=det, modes=modes, bins=size(192, 378),
                    phases=min(phases, 32), snr=snr, precision=rng.choice(["mixed", "fp16x3"]), cut=CUT)
    if kind == "precessing":
        return dict(kind="precessing", rows=size(2048, 16384), ext=size(256, 4096), det=det, modes=modes, bins=bins,
                    phases=phases, snr=snr, precision="mixed", cut=CUT)
    if kind == "presel":
        return dict(kind="presel", rows=size(2048, 65536), times=rng.choice([64, 100, 128]), det=det, modes=modes, bins=bins,
                    phases=min(phases, 32), snr=snr, precision=rng.choice(["fp16x3", "bf16x3"]))
    if kind == "presel_pol":
        return dict(kind="presel_pol", rows=size(1024, 16384), times=rng.choice([64, 100, 128]), det=det, modes=modes,
                    bins=size(192, 378), phases=min(phases, 32), snr=snr, precision="fp32")
    return dict(kind="samples", rows=size(2048, 16384), ext=size(256, 2048), det=det, modes=modes, bins=bins,
                phases=min(phases, 32), snr=snr, draws=size(32, 512))


# ---- inputs ------------------------------------------------------------------------------------------------------
def _grid(bins, fmin=20.0, fmax=1024.0):
    f = fmin * (fmax / fmin) ** (np.arange(bins) / (bins - 1))
    return f, _trapezoid(f)


def _trapezoid(f):
    w = np.empty(f.shape[0])
    w[0], w[-1] = 0.5 * (f[1] - f[0]), 0.5 * (f[-1] - f[-2])
    w[1:-1] = 0.5 * (f[2:] - f[:-2])
    return w


def _psd(f, det):
    r = f / 150.0
    return np.stack([s * (r ** -4 + 2.0 + 2.0 * r ** 2) for s in PSD_SCALE[:det]])


def _pol(l, m, iota):
    """(K+, Kx / i) of a mode at inclination iota (both real): spin-weight -2 harmonics at azimuth 0."""
    c, s, ci, si = torch.cos(iota / 2), torch.sin(iota / 2), torch.cos(iota), torch.sin(iota)
    if (l, m) == (2, 2):
        n = math.sqrt(5 / (64 * math.pi))
        yp, ym = n * (1 + ci) ** 2, n * (1 - ci) ** 2
    elif (l, m) == (2, 1):
        n = math.sqrt(5 / (16 * math.pi))
        yp, ym = n * si * (1 + ci), n * si * (1 - ci)
    elif (l, m) == (3, 3):
        n = math.sqrt(21 / (2 * math.pi))
        yp, ym = -n * c ** 5 * s, n * c * s ** 5
    else:
        n = 3 * math.sqrt(7 / math.pi)
        yp, ym = n * c ** 6 * s ** 2, n * c ** 2 * s ** 6
    sign = (-1.0) ** l
    return 0.5 * (yp + sign * ym), 0.5 * (yp - sign * ym)


def _pol_np(l, m, iota):
    kp, kx = _pol(l, m, torch.as_tensor(iota, dtype=torch.float64))
    return kp.numpy().astype(complex), 1j * kx.numpy()


def _waveforms(f, mc, ratios, mode_m, amp22, wobble=None, modes=None, dtype=torch.complex64, device="cuda"):
    """h [rows, M, B], or [rows, M, 2, B] with each row's inclination wobbling along the frequency."""
    t = lambda x: torch.as_tensor(np.asarray(x, dtype=np.float64), device=device)  # noqa: E731
    f, mc, ratios, amp22 = t(f), t(mc), t(ratios), t(amp22)
    rows, M, B = mc.shape[0], len(mode_m), f.shape[0]
    shape = (rows, M, B) if wobble is None else (rows, M, 2, B)
    out = torch.empty(shape, dtype=dtype, device=device)
    base = f ** (-7 / 6)
    step = max(1, (1 << 23) // B)
    for r0 in range(0, rows, step):
        r1 = min(rows, r0 + step)
        x = math.pi * GM_SUN_S * mc[r0:r1, None] * f
        psi22 = -0.25 * math.pi + (3 / 128) * x ** (-5 / 3)
        if wobble is not None:
            i0, am, pe = (t(v[r0:r1])[:, None] for v in wobble)
            iota = i0 + am * torch.sin(2 * math.pi * torch.log(f / f[0]) / pe)
        for k, m in enumerate(mode_m):
            h = torch.polar((amp22[r0:r1] * ratios[r0:r1, k])[:, None] * base, (0.5 * int(m)) * psi22)
            if wobble is None:
                out[r0:r1, k] = h
            else:
                kp, kx = _pol(*modes[k], iota)
                out[r0:r1, k, 0] = kp * h
                out[r0:r1, k, 1] = 1j * kx * h
    return out


def _extrinsic(lat, lon, psi, cos_iota, t_geo, det, modes):
    """Arrival times t [E, D], mode responses R [E, D, M] and antenna patterns F [E, D, 2]."""
    src = np.stack([np.cos(lat) * np.cos(lon), np.cos(lat) * np.sin(lon), np.sin(lat)], -1)
    th, ph = 0.5 * np.pi - lat, lon
    X = np.stack([np.sin(ph) * np.cos(psi) - np.sin(psi) * np.cos(ph) * np.cos(th),
                  -(np.cos(ph) * np.cos(psi) + np.sin(psi) * np.sin(ph) * np.cos(th)), np.sin(psi) * np.sin(th)], -1)
    Y = np.stack([-np.sin(ph) * np.sin(psi) - np.cos(psi) * np.cos(ph) * np.cos(th),
                  np.cos(ph) * np.sin(psi) - np.cos(psi) * np.sin(ph) * np.cos(th), np.cos(psi) * np.sin(th)], -1)
    K = [_pol_np(l, m, np.arccos(cos_iota)) for l, m in modes]
    E = lat.shape[0]
    t, R, F = np.empty((E, det)), np.empty((E, det, len(modes)), complex), np.empty((E, det, 2))
    for d, (la, lo, xa, ya) in enumerate(SITES[:det]):
        la, lo = math.radians(la), math.radians(lo)
        r = np.array([math.cos(la) * math.cos(lo), math.cos(la) * math.sin(lo), math.sin(la)])
        east = np.array([-math.sin(lo), math.cos(lo), 0.0])
        north = np.array([-math.sin(la) * math.cos(lo), -math.sin(la) * math.sin(lo), math.cos(la)])
        x, y = (math.cos(math.radians(b)) * north + math.sin(math.radians(b)) * east for b in (xa, ya))
        T = 0.5 * (np.outer(x, x) - np.outer(y, y))
        q = lambda a, b: np.einsum("ni,ij,nj->n", a, T, b)  # noqa: E731
        F[:, d, 0], F[:, d, 1] = q(X, X) - q(Y, Y), q(X, Y) + q(Y, X)
        t[:, d] = t_geo - R_EARTH * (src @ r) / C_LIGHT
        for k, (kp, kx) in enumerate(K):
            R[:, d, k] = F[:, d, 0] * kp + F[:, d, 1] * kx
    return t, R, F


def _prior(rng, n):
    lon, lat = rng.uniform(0, 2 * np.pi, n), np.arcsin(rng.uniform(-1, 1, n))
    return lat, lon, rng.uniform(0, np.pi, n), rng.uniform(-1, 1, n), rng.uniform(-0.01, 0.01, n)


def _noise(rng, psd, w):
    return np.sqrt(psd / (4 * w)) * (rng.standard_normal(psd.shape) + 1j * rng.standard_normal(psd.shape))


def _signal(h, r, t, f, mode_m, phi):
    """sum_j h_j r_dj e^{i m_j phi} shifted to each detector; h [J, B], r [D, J], mode_m [J]."""
    return np.einsum("jb,dj,j->db", h, r, np.exp(1j * mode_m * phi)) * np.exp(-2j * np.pi * f * t[:, None])


class _Inputs:
    """One event's inputs and the bank they go with (host arrays; h on the GPU)."""

    def __init__(self, c, seed):
        self.c = c
        kind = c["kind"]
        rng = self.rng = np.random.default_rng(int(seed))
        self.modes = MODES[c["modes"]]
        self.mode_m = np.array([m for _, m in self.modes], dtype=np.int32)
        self.rb = kind in ("rb", "presel_pol")
        self.pol = kind in ("precessing", "presel_pol")
        M = len(self.modes)
        i22 = self.modes.index((2, 2))
        n_bank = c.get("bank", c.get("rows"))
        det = c.get("det", 3)
        if self.rb:
            self.f_fine = np.linspace(20.0, 1024.0, N_FINE)
            self.df = np.full(N_FINE, self.f_fine[1] - self.f_fine[0])
            self.df[[0, -1]] *= 0.5
            at = _grid(c["bins"])[0]
            self.nodes = np.clip(np.rint((at - 20.0) / (self.f_fine[1] - self.f_fine[0])).astype(np.int64), 0, N_FINE - 1)
            self.f = self.f_fine[self.nodes]
            self.w = _trapezoid(self.f)
            self.psd_fine = _psd(self.f_fine, det)
            mc0 = 12.0
            mc = mc0 * (1 + rng.uniform(-0.02, 0.02, n_bank))
            mc[0] = mc0
            norm = math.sqrt(np.sum(4 * self.df * self.f_fine ** (-7 / 3) / self.psd_fine[0]))
        else:
            self.f, self.w = _grid(c["bins"])
            mc0 = 17.5
            mc = rng.uniform(5.0, 30.0, n_bank)
            norm = math.sqrt(np.sum(4 * self.w * self.f ** (-7 / 3) / _psd(self.f, 1)[0]))
        ratios = rng.uniform(0.0, 0.3, (n_bank, M))
        if self.rb:
            ratios[0] = rng.uniform(0.05, 0.3, M)
        ratios[:, i22] = 1.0
        amp22 = (mc / mc0) ** (5 / 6) / norm
        wob = None
        if self.pol:
            wob = (np.arccos(rng.uniform(-1, 1, n_bank)), rng.uniform(0, 0.5, n_bank), rng.uniform(0.5, 2.0, n_bank))
        self.wave = dict(mode_m=self.mode_m, modes=self.modes)
        self.rows_of = lambda k: dict(mc=mc[k], ratios=ratios[k], amp22=amp22[k],  # noqa: E731
                                      wobble=None if wob is None else tuple(v[k] for v in wob))
        self.h = _waveforms(self.f, **self.rows_of(slice(None)), **self.wave)
        self.ln_w_int = np.zeros(n_bank)
        self.i0, self.i1 = 0, n_bank
        if kind == "event" and c["rows"] < n_bank:
            self.i0 = int(rng.integers(0, n_bank - c["rows"] + 1))
            self.i1 = self.i0 + c["rows"]
        if kind == "event" and c["cut"] == 0:
            self.ln_w_int = rng.normal(0.0, 0.5, n_bank)
        self.j_m = np.repeat(self.mode_m, 2) if self.pol else self.mode_m
        if kind == "batch":
            # extrinsic counts over a factor of eight, two or three detectors, quiet and loud: the same mix at every seed
            mix = np.random.default_rng(c["events"])
            self.events = [self._event(det=int(mix.integers(2, 4)), n_ext=int(c["ext"] * mix.uniform(0.22, 1.78)),
                                       snr=float(mix.uniform(8, 40))) for _ in range(c["events"])]
        else:
            self.events = [self._event(det=det, n_ext=c.get("ext", 1), snr=c["snr"])]

    def _event(self, det, n_ext, snr):
        rng, e = self.rng, {}
        lat, lon, psi, ci, tg = _prior(rng, 1)
        t1, R1, F1 = _extrinsic(lat, lon, psi, ci, tg, det, self.modes)
        phi = rng.uniform(0, 2 * np.pi)
        inj = 0 if self.rb else int(rng.integers(self.i0, self.i1))
        f = self.f_fine if self.rb else self.f
        w = self.df if self.rb else self.w
        psd = _psd(f, det)
        h = _waveforms(f, **{k: (None if v is None else tuple(x[None] for x in v) if k == "wobble" else np.asarray(v)[None])
                             for k, v in self.rows_of(inj).items()}, **self.wave, dtype=torch.complex128, device="cpu")
        h = h.numpy()[0].reshape(len(self.j_m), -1)
        r = np.tile(F1[0], (1, len(self.modes))) if self.pol else R1[0]
        s = _signal(h, r, t1[0], f, self.j_m, phi)
        s *= snr / math.sqrt(np.sum(4 * w * np.abs(s) ** 2 / psd))
        data = s + _noise(rng, psd, w)
        if self.rb:
            e.update(psd_fine=psd, data_fine=data, h0=h, t0=t1[0].copy())
            ext = (np.clip(lat + rng.normal(0, 0.05, n_ext), -np.pi / 2, np.pi / 2), lon + rng.normal(0, 0.05, n_ext),
                   rng.uniform(0, np.pi, n_ext), rng.uniform(-1, 1, n_ext), tg + rng.normal(0, 5e-4, n_ext))
        else:
            e.update(psd=psd, data=data)
            ext = _prior(rng, n_ext)
        e["t"], e["R"], e["F"] = _extrinsic(*ext, det, self.modes)
        e["det"], e["inj"], e["cos_iota"] = det, inj, float(ci[0])
        e["ln_w_ext"] = rng.normal(0, 0.5, n_ext) if self.c.get("cut") == 0 else np.zeros(n_ext)
        kp = abs(_pol_np(2, 2, np.zeros(1))[0][0])
        e["u_min"] = 4.0 / math.sqrt(sum(kp ** 2 / s for s in PSD_SCALE[:det]))
        return e

    def presel_extra(self):
        """The time grid, and each row's polarisation factors (the inclination is the row's own there)."""
        c, rng = self.c, self.rng
        ci = rng.uniform(-1, 1, self.h.shape[0])
        ci[self.events[0]["inj"]] = self.events[0]["cos_iota"]
        K = np.empty((self.h.shape[0], len(self.modes), 2), complex)
        for k, (l, m) in enumerate(self.modes):
            K[:, k, 0], K[:, k, 1] = _pol_np(l, m, np.arccos(ci))
        return K, np.tile((np.arange(c["times"]) - c["times"] // 2) * 5e-4, (c["det"], 1))


# ---- what a user's program keeps, and one pass -------------------------------------------------------------------
class _State:
    """A context, its bank and the inputs of the next call; gives them back at the end."""

    def __init__(self, case):
        self.case, self.ctx, self.bank, self.event = case, dp.dotpe_create(0), None, None

    def __del__(self):
        if self.event is not None:
            dp.dotpe_event_release(self.ctx, self.event)
        dp.dotpe_destroy(self.ctx)


def prepare(case, seed):
    c = case
    x = _Inputs(c, seed)
    s = _State(c)
    kind = c["kind"]
    pol = None
    if kind == "presel":
        pol, s.t_grid = x.presel_extra()
    elif kind == "presel_pol":
        _, s.t_grid = x.presel_extra()
    torch.cuda.synchronize()
    s.bank = dp.dotpe_bank_load(s.ctx, x.h, x.f, x.w, x.mode_m, x.ln_w_int, pol)
    dev = (lambda a: a) if c.get("host", kind == "rb") else (lambda a: torch.as_tensor(a, device="cuda"))
    s.calls = []
    for e in x.events:
        call = dict(bank_id=s.bank, i0=x.i0, i1=x.i1, psd=None, data=None, t=dev(e["t"]), R=dev(e["R"]),
                    ln_w_ext=dev(e["ln_w_ext"]) if c.get("cut") == 0 else None, n_phi=c["phases"], u_min=e["u_min"],
                    cut_delta=c.get("cut", CUT), precision=c.get("precision", "mixed"), block_rows=c.get("block", 0),
                    flags=dp.DOTPE_FLAG_STORE_LNL if c.get("store") or kind == "samples" else 0)
        if kind == "precessing":
            call.update(F=dev(e["F"]), R=None)
        if not x.rb:
            call.update(psd=dev(e["psd"]), data=dev(e["data"]))
        s.calls.append(call)
    e = x.events[0]
    if x.rb:
        s.fine = (x.f_fine, x.df, e["psd_fine"], e["data_fine"], e["h0"], x.nodes, e["t0"])
    if kind == "presel":
        s.presel = dict(psd=e["psd"], data=e["data"])
    elif kind == "presel_pol":
        s.presel = dict(psd=None, data=None, rb=dp.dotpe_rb_weights(s.ctx, *s.fine))
    elif kind == "samples":
        s.event = dp.dotpe_event_submit(s.ctx, **s.calls[0])
        dp.dotpe_event_wait(s.ctx, s.event)
        s.uniforms = x.rng.uniform(size=(c["draws"], 4))
    torch.cuda.synchronize()
    return s


def _marginal(s, eid, what, n):
    out = torch.empty(n, dtype=torch.float32, device="cuda")
    row = what == dp.DOTPE_ROW_MARGINAL
    return dp.dotpe_lnl_blocks(s.ctx, eid, 0, n if row else 1, 0, 1 if row else n, what, out)


def _results(s, call, eid):
    """What a program reads of a finished event: the evidence, the marginals, and the stored pairs where it asked for them."""
    dp.dotpe_event_wait(s.ctx, eid)
    ev = dp.dotpe_evidence(s.ctx, eid)
    NI, NE = call["i1"] - call["i0"], call["t"].shape[0]
    out = {"ln_z": ev["ln_z"], "max_lnl_ml": ev["max_lnl_ml"]}
    block = lambda what: dp.dotpe_lnl_blocks(s.ctx, eid, 0, NI, 0, NE, what,  # noqa: E731
                                             torch.empty(NI, NE, dtype=torch.float32, device="cuda"))
    if call["precision"] != "fp32" and not (call["precision"] != "mixed" and call["cut_delta"] > 0):
        # (a running cut keeps a set of pairs that differs by a few from run to run, and with it the marginals' tails)
        out["ln_p_ext"] = _marginal(s, eid, dp.DOTPE_COL_MARGINAL, NE)
    if call["cut_delta"] == 0:
        out["ln_p_int"] = _marginal(s, eid, dp.DOTPE_ROW_MARGINAL, NI)
        out["lnl"] = block(dp.DOTPE_LNL_MARG)
    if call["flags"] & dp.DOTPE_FLAG_STORE_LNL:
        out["lnl_ml"] = block(dp.DOTPE_LNL_ML_MAX)
    dp.dotpe_event_release(s.ctx, eid)
    return out


def run(state):
    s = state
    kind = s.case["kind"]
    if kind in ("event", "precessing"):
        return _results(s, s.calls[0], dp.dotpe_event_submit(s.ctx, **s.calls[0]))
    if kind == "batch":
        return [_results(s, c, e) for c, e in zip(s.calls, dp.dotpe_batch_submit(s.ctx, s.calls))]
    if kind == "rb":
        w = dp.dotpe_rb_weights(s.ctx, *s.fine)
        return {"w_dh": w[0], "w_hh": w[1], **_results(s, s.calls[0], dp.dotpe_event_submit(s.ctx, rb=w, **s.calls[0]))}
    if kind in ("presel", "presel_pol"):
        r = dp.dotpe_preselect(s.ctx, s.bank, 0, s.case["rows"], t_grid=s.t_grid, n_phi=s.case["phases"], delta=CUT,
                               precision=s.case["precision"], outputs=("lnl_ml", "selected"), **s.presel)
        keep = np.zeros(s.case["rows"], dtype=bool)
        keep[r["selected"]] = True
        return {"lnl_ml": r["lnl_ml"], "keep": keep, "max_lnl_inco": r["max_lnl_inco"]}
    i, e, o, d = dp.dotpe_posterior_samples(s.ctx, s.event, s.uniforms)
    return {"i": i, "e": e, "o": o, "distance": d}


def work(case):
    c, kind = case, case["kind"]
    M, B, D = c["modes"], c["bins"], c.get("det", 3)
    P = 2 if kind in ("precessing", "presel_pol") else 1
    rows = c.get("rows", c.get("bank"))
    # the bank's operand as the precision holds it: FP32, one 16-bit plane for a screen, two for a split product
    el = {"fp32": 4, "mixed": 2}.get(c.get("precision", "mixed"), 4)
    bank = rows * M * P * 2 * B * el
    if kind in ("presel", "presel_pol"):
        cols = D * c["times"]
        return {"bytes": bank + rows * D * 4, "flops": float(rows) * cols * (8 * M * P * B + c["phases"] * (4 * M * 2 + 6))}
    if kind == "samples":
        # per draw: one row of stored values, the pair in 64 bits over the bins
        n = c["draws"]
        return {"bytes": rows * 8 + n * (c["ext"] * 4 + 8 * M * B), "flops": float(n) * D * B * (16 * M + 8 * M * (M + 1) / 2)}
    pair = 8 * M * P * B + (42 * D if P == 2 else D * (2 * M + 4 * M * (M - 1)))
    n_ext = c["ext"] * (c["events"] if kind == "batch" else 1)
    b = bank + n_ext * D * (8 + 16 * M) + n_ext * 4
    if c.get("store"):
        b += rows * c["ext"] * 4 * (2 if c["cut"] == 0 else 1)
    f = float(rows) * n_ext * pair
    if c.get("cut") == 0 or c.get("precision") == "fp32":
        f += float(rows) * n_ext * c["phases"] * (4 * M + 14)  # the phase grid of every pair
    if kind == "rb":
        b += N_FINE * (16 + D * 24 + M * 16)
        f += float(N_FINE) * D * 2 * (8 * M + 8 * M * (M + 1) / 2)
    return {"bytes": b, "flops": f}


# ---- 64-bit values -----------------------------------------------------------------------------------------------
_GL = {n: tuple(torch.as_tensor(v) for v in np.polynomial.legendre.leggauss(n)) for n in (48, 144)}


def _ln_lbar(dh, hh, u_min):
    """ln of 3 u^3 int_u^inf v^-4 exp(dh v - hh v^2 / 2) dv: Gauss-Legendre in ln v, below the peak and over it."""
    r = torch.sqrt(hh)
    x, s = dh / r, u_min * r
    top = torch.maximum(x, s) + 9.0
    mid = torch.maximum(s, x - 8.0)
    out = torch.zeros_like(x)
    for lo, hi, n in ((s, mid, 48), (mid, top, 144)):
        z, g = (v.to(x.device) for v in _GL[n])
        half = 0.5 * (torch.log(hi) - torch.log(lo))
        ln_v = torch.log(lo)[:, None] + half[:, None] * (z + 1)
        v = torch.exp(ln_v)
        # scaled by the largest value of exp(x v - v^2 / 2) on [s, inf)
        peak = torch.maximum(x, s)[:, None]
        ex = (x[:, None] - 0.5 * (v + peak)) * (v - peak) - 3 * (ln_v - torch.log(s)[:, None])
        out += half * (torch.exp(ex) @ g)
    peak = torch.maximum(x, s)
    return math.log(3.0) + torch.log(out) + (x - 0.5 * peak) * peak


def _lse_by(index, n, v):
    """ln sum exp(v) per index; -inf where there is none."""
    m = torch.full((n,), -math.inf, dtype=v.dtype, device=v.device).scatter_reduce(0, index, v, "amax")
    s = torch.zeros(n, dtype=v.dtype, device=v.device).index_add_(0, index, torch.exp(v - m[index]))
    return m + torch.log(s)


def _rb_exact(x, e):
    """The weights of relative binning by their sums over the fine grid."""
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    f, df, psd, data = dev(x.f_fine), dev(x.df), dev(e["psd_fine"]), dev(e["data_fine"])
    nodes, h0, t0 = dev(x.nodes), dev(e["h0"]), dev(e["t0"])
    B, D, J = nodes.shape[0], psd.shape[0], h0.shape[0]
    n = torch.arange(int(nodes[0]), int(nodes[-1]) + 1, device="cuda")
    b = torch.clamp(torch.searchsorted(nodes, n, right=True) - 1, max=B - 2)
    up = (f[n] - f[nodes[b]]) / (f[nodes[b + 1]] - f[nodes[b]])
    w_dh = torch.empty(D, J, B, dtype=torch.complex128, device="cuda")
    w_hh = torch.empty(D, J, J, B, dtype=torch.complex128, device="cuda")

    def hat(v):  # sums against the hat functions
        z = torch.zeros(B, dtype=v.dtype, device="cuda")
        return z.index_add(0, b, v * (1 - up)).index_add(0, b + 1, v * up)

    for d in range(D):
        h = h0 * torch.exp(-2j * math.pi * f * t0[d])
        w = 4 * df / psd[d]
        for j in range(J):
            w_dh[d, j] = hat((w * data[d] * h[j].conj())[n]) / h[j, nodes].conj()
            for k in range(J):
                w_hh[d, j, k] = hat((w * h[j] * h[k].conj())[n]) / (h[j, nodes] * h[k, nodes].conj())
    return w_dh, w_hh


class _Pairs:
    """Z_m and the coefficients of <h|h> of bank rows against one event's samples, in 64 bits."""

    def __init__(self, x, e, w=None):
        dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
        self.x, self.M, P = x, len(x.modes), 2 if x.pol else 1
        f, t = dev(x.f), dev(e["t"])
        D, E, J = t.shape[1], t.shape[0], self.M * P
        if w is None:
            om = 4 * dev(x.w) / dev(e["psd"])
            c = (om * dev(e["data"]).conj())[:, None].expand(D, J, -1)
            self.om = om[:, None, None].expand(D, J, J, -1)
        else:
            c, self.om = w[0].conj(), w[1]
        r = dev(e["F"]).repeat(1, 1, self.M).to(torch.complex128) if x.pol else dev(e["R"])  # [E, D, J]
        self.G = torch.zeros(self.M, P * len(x.f), E, dtype=torch.complex128, device="cuda")
        for d in range(D):
            T = torch.exp(-2j * math.pi * f[:, None] * t[:, d])
            for j in range(J):
                self.G[j // P, (j % P) * len(x.f):(j % P + 1) * len(x.f)] += r[:, d, j] * T * c[d, j][:, None]
        self.delta = sorted({int(a - b) for a in x.j_m for b in x.j_m if a >= b})
        self.q = {dl: [] for dl in self.delta}  # (d, j, k) and the samples' factors r_j r_k^*
        for dl in self.delta:
            at = [(d, j, k) for d in range(D) for j in range(J) for k in range(J) if x.j_m[j] - x.j_m[k] == dl]
            self.q[dl] = (at, torch.stack([r[:, d, j] * r[:, d, k].conj() for d, j, k in at]))
        o = torch.arange(x.c["phases"], device="cuda", dtype=torch.float64) * (2 * math.pi / x.c["phases"])
        self.phase = lambda m: torch.exp(1j * m * o)  # noqa: E731

    def of_rows(self, i0, i1):
        h = self.x.h[i0:i1].to(torch.complex128)
        Z = torch.stack([h[:, m].reshape(i1 - i0, -1) @ self.G[m] for m in range(self.M)])
        hj = h.reshape(i1 - i0, len(self.x.j_m), -1)
        C = torch.stack([torch.stack([((hj[:, j] * hj[:, k].conj()) @ self.om[d, j, k].to(torch.complex128)) for d, j, k in self.q[dl][0]], 1)
                         @ self.q[dl][1] for dl in self.delta])
        return Z, C

    def on_phases(self, Z, C):
        """dh, hh [n, n_phi] of n pairs; Z [M, n], C [len(delta), n]."""
        dh = sum((Z[m][:, None] * self.phase(int(self.x.mode_m[m]))).real for m in range(self.M))
        hh = sum((C[k][:, None] * self.phase(dl)).real * (1.0 if dl == 0 else 2.0) for k, dl in enumerate(self.delta))
        return dh, hh


def _ml(dh, hh):
    return torch.where((dh > 0) & (hh > 0), 0.5 * dh * dh / hh, torch.zeros_like(dh))


def _event_exact(x, e, w=None, want_ml=False):
    """ln Z, max ln L^ML, marginals and (without a cut) ln Lbar of every pair."""
    c = x.c
    p = _Pairs(x, e, w)
    NI, NE, cut, np_ = x.i1 - x.i0, e["t"].shape[0], c["cut"], c["phases"]
    lwi = torch.as_tensor(x.ln_w_int[x.i0:x.i1], device="cuda")
    lwe = torch.as_tensor(e["ln_w_ext"], device="cuda")
    step = max(1, min(NI, (1 << 22) // NE))
    best, kept, ml_all, lnl_all = 0.0, [], [], []
    for r0 in range(0, NI, step):
        r1 = min(NI, r0 + step)
        Z, C = (v.reshape(v.shape[0], -1) for v in p.of_rows(x.i0 + r0, x.i0 + r1))
        at = torch.arange(Z.shape[1], device="cuda")
        if cut > 0 and not want_ml:
            # pairs that can reach the cut: |dh| <= sum |Z_m|, hh >= C_0 - 2 sum |C_delta|
            lo = C[0].real - 2 * C[1:].abs().sum(0)
            top = torch.where(lo > 0, 0.5 * Z.abs().sum(0) ** 2 / lo.clamp_min(1e-300), math.inf)
            first = torch.topk(top, min(256, top.shape[0])).indices
            best = max(best, float(_ml(*p.on_phases(Z[:, first], C[:, first])).max()))
            at = torch.nonzero(top >= best - cut)[:, 0]
        rows_ml, rows_l = [], []
        for a in torch.split(at, 1 << 18) if at.numel() else ():
            dh, hh = p.on_phases(Z[:, a], C[:, a])
            ml = _ml(dh, hh)
            best = max(best, float(ml.max()))
            if want_ml or cut == 0:
                rows_ml.append(ml.max(1).values)
            if cut == 0:
                l = torch.cat([_ln_lbar(u, v, e["u_min"]) for u, v in zip(torch.split(dh.reshape(-1), 1 << 20), torch.split(hh.reshape(-1), 1 << 20))])
                rows_l.append(torch.logsumexp(l.reshape(dh.shape), 1))
            else:
                n, o = torch.nonzero(ml >= best - cut, as_tuple=True)
                kept.append((a[n] // NE + r0, a[n] % NE, dh[n, o], hh[n, o], ml[n, o]))
        if rows_ml:
            ml_all.append(torch.cat(rows_ml).reshape(r1 - r0, NE))
        if rows_l:
            lnl_all.append(torch.cat(rows_l).reshape(r1 - r0, NE))
    out = {"max_lnl_ml": best}
    if cut == 0:
        lnl = torch.cat(lnl_all)
        v = lnl + lwi[:, None] + lwe
        out["ln_p_int"], out["ln_p_ext"] = torch.logsumexp(v, 1), torch.logsumexp(v, 0)
        out["lnl"] = lnl - math.log(np_)
        total = torch.logsumexp(v.reshape(-1), 0)
    else:
        i, k, dh, hh, ml = (torch.cat(q) for q in zip(*kept))
        g = ml >= best - cut
        i, k = i[g], k[g]
        l = torch.cat([_ln_lbar(u, v, e["u_min"]) for u, v in zip(torch.split(dh[g], 1 << 20), torch.split(hh[g], 1 << 20))])
        out["ln_p_ext"] = _lse_by(k, NE, l + lwi[i] + lwe[k])
        total = torch.logsumexp(l + lwi[i] + lwe[k], 0)
    if ml_all:
        out["lnl_ml"] = torch.cat(ml_all)
    out["ln_z"] = float(total) - math.log(NI) - math.log(NE) - math.log(np_)
    return {k: np.float64(v) if isinstance(v, float) else v for k, v in out.items()}


def _presel_exact(x, e):
    """max over (phase, time) of the single-detector ln L^ML with both polarisation amplitudes free."""
    dev = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    K, t_grid = x.presel_extra()
    f, M, np_ = dev(x.f), len(x.modes), x.c["phases"]
    D, rows = x.c["det"], x.h.shape[0]
    w = _rb_exact(x, e) if x.rb else None
    if w is None:
        om = 4 * dev(x.w) / dev(e["psd"])
        cw = om * dev(e["data"]).conj()
    o = torch.arange(np_, device="cuda", dtype=torch.float64) * (2 * math.pi / np_)
    ph = [torch.exp(1j * int(m) * o) for m in x.mode_m]
    out = torch.empty(rows, D, dtype=torch.float64, device="cuda")
    K = dev(K)
    for d in range(D):
        T = torch.exp(-2j * math.pi * f[:, None] * dev(t_grid[d]))
        for r0 in range(0, rows, 2048):
            r1 = min(rows, r0 + 2048)
            h = x.h[r0:r1].to(torch.complex128)
            hp = h if x.pol else K[r0:r1, :, :, None] * h[:, :, None]  # [n, M, 2, B]
            if w is None:
                Zj = [[(hp[:, m, p] @ (cw[d][:, None] * T)) for p in range(2)] for m in range(M)]
                O = lambda a, p, b, q: (hp[:, a, p] * hp[:, b, q].conj()) @ om[d].to(torch.complex128)  # noqa: E731
            else:
                Zj = [[hp[:, m, p] @ (w[0][d, 2 * m + p].conj()[:, None] * T) for p in range(2)] for m in range(M)]
                O = lambda a, p, b, q: (hp[:, a, p] * hp[:, b, q].conj()) @ w[1][d, 2 * a + p, 2 * b + q]  # noqa: E731
            H = {}
            for p, q in ((0, 0), (0, 1), (1, 1)):
                H[p, q] = sum((O(a, p, b, q)[:, None] * (ph[a] * ph[b].conj())).real for a in range(M) for b in range(M))
            A, X, Cc = H[0, 0], H[0, 1], H[1, 1]
            det = A * Cc - X * X
            inv = det > 1e-3 * A * Cc
            ia = torch.where(inv, Cc / det, A / (A + Cc) ** 2)
            ic = torch.where(inv, A / det, Cc / (A + Cc) ** 2)
            ix = torch.where(inv, -X / det, X / (A + Cc) ** 2)
            best = torch.zeros(r1 - r0, dtype=torch.float64, device="cuda")
            for k in range(np_):
                u, v = (sum((Zj[m][p] * ph[m][k]).real for m in range(M)) for p in range(2))
                val = 0.5 * (ia[:, k, None] * u * u + 2 * ix[:, k, None] * u * v + ic[:, k, None] * v * v)
                best = torch.maximum(best, val.max(1).values)
            out[r0:r1, d] = best
    return {"lnl_ml": out, "keep": None, "max_lnl_inco": np.float64(float(out.sum(1).max()))}


def exact(case, seed):
    kind = case["kind"]
    if kind == "samples":
        return None  # whole numbers, and draws that follow from them
    x = _Inputs(case, seed)
    if kind in ("presel", "presel_pol"):
        return _presel_exact(x, x.events[0])
    if kind == "batch":
        got = [_event_exact(x, e) for e in x.events]
    else:
        w = _rb_exact(x, x.events[0]) if x.rb else None
        got = [_event_exact(x, x.events[0], w, want_ml=bool(case.get("store")))]
        if w is not None:
            got[0].update(w_dh=w[0], w_hh=w[1])
        if not case.get("store") or case["precision"] == "fp32":
            got[0].pop("lnl", None)
        if case["precision"] == "fp32" or (case["precision"] != "mixed" and case["cut"] > 0):
            got[0].pop("ln_p_ext", None)
    return got if kind == "batch" else got[0]
