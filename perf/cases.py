"""Performance cases of the ratio-filter library, through its public Python calls.

Every input is drawn from a seed: strain with an aLIGO-like noise colour, stored filters and
templates of 1-3 solar-mass inspirals, and ratio kernels that are the windowed, truncated
chirps of a neighbour's phase difference, imported as a search imports its stored kernels.
Sizes follow the library's workloads: n = 2^16 at 1024 Hz, n = 2^20 (512 s) and n = 2^23
(4096 s) at 2048 Hz, with 16, 256 and 128 neighbours per reference.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_12894_gb300 import RatioFilter

MSUN_S = 4.925491025543576e-6   # G M_sun / c^3 in seconds
DF_HIGH, DF_LOW_MAX = 53.0, 5.0  # the library's default taper widths (Hz)
THRESHOLD = 3e-5                 # relative truncation threshold of the benchmark

# Layouts of the batched and single-reference peaks, as "cut:block:part[:form]" per length bucket;
# "" leaves the choice to the library.
TWO = "0:4096:1024,4096:16384:4096"
THREE = "0:16384:4096,8192:16384:8192,65536:32768:16384:os_bins"


def listed():
    return [
        # -- reference matched filters
        # the smallest call: one stored filter over a 16 s segment, as a low-latency loop makes it
        dict(name="mf_small", kind="mf", n=1 << 14, fs=1024.0, f_low=40.0, dtype="f32", refs=1, W=0),
        # the double-precision check path: templates generated in the call
        dict(name="mf_f64", kind="mf_ref", n=1 << 16, fs=1024.0, f_low=40.0, dtype="f64", refs=1, pn=2),
        # waveform generation plus correlation, the paper's standard method, single precision
        dict(name="mf_onthefly", kind="mf_ref", n=1 << 20, fs=2048.0, f_low=20.0, dtype="f32", refs=3, pn=7),
        # the references of a batched search over one segment, with their peaks per minute
        dict(name="mf_bank", kind="mf", n=1 << 20, fs=2048.0, f_low=20.0, dtype="f32", refs=24, W=1 << 17),
        # the long-duration search's references (4096 s segments)
        dict(name="mf_long", kind="mf", n=1 << 23, fs=2048.0, f_low=5.0, dtype="f32", refs=6, W=1 << 20),
        # -- neighbours' series and peaks from the reference's series
        # full series of a few neighbours (follow-up of a candidate), the library's own layout
        dict(name="series", kind="recon", n=1 << 18, fs=2048.0, f_low=20.0, dtype="f32", refs=1, k=21,
             tau0=0.05, tau1=3.0, W=0, algo="auto", prec="native", real=False, layout=""),
        # the paper-shaped set: one reference, 256 neighbours, peaks per minute, two length buckets
        dict(name="peaks", kind="recon", n=1 << 20, fs=2048.0, f_low=20.0, dtype="f32", refs=1, k=256,
             tau0=0.05, tau1=15.0, W=1 << 17, algo="auto", prec="native", real=False, layout=TWO),
        # several references in one call with real-form kernels (half the stored bytes)
        dict(name="peaks_real", kind="recon", n=1 << 20, fs=2048.0, f_low=20.0, dtype="f32", refs=3, k=32,
             tau0=0.05, tau1=15.0, W=1 << 18, algo="auto", prec="native", real=True, layout=TWO),
        # the long-duration search: kernels up to 2.6e5 taps in three length buckets
        dict(name="peaks_long", kind="recon", n=1 << 23, fs=2048.0, f_low=5.0, dtype="f32", refs=2, k=48,
             tau0=0.05, tau1=120.0, W=1 << 20, algo="auto", prec="native", real=False, layout=THREE),
        # the double-precision check path of the reconstruction
        dict(name="peaks_f64", kind="recon", n=1 << 16, fs=1024.0, f_low=40.0, dtype="f64", refs=1, k=16,
             tau0=0.002, tau1=0.05, W=1024, algo="auto", prec="native", real=False, layout=""),
        # short kernels on the tensor cores at FP32-equivalent accuracy
        dict(name="peaks_tensor", kind="recon", n=1 << 16, fs=1024.0, f_low=40.0, dtype="f32", refs=1, k=16,
             tau0=0.002, tau1=0.05, W=1024, algo="gemm", prec="bf16x6", real=False, layout=""),
        # -- making the ratio kernels of a reference's neighbours (once per bank and noise curve)
        dict(name="build", kind="build", n=1 << 19, fs=2048.0, f_low=20.0, dtype="f32", k=48, pn=7, spread=0.01,
             n_build=0, real=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: any segment length between the listed ones, odd counts,
    ragged last windows, both kernel forms, both grids."""
    kind = rng.choice(["mf", "mf_ref", "recon", "recon", "recon", "build"])
    if kind == "mf":
        b = rng.randint(14, 23)
        low = b > 21
        n = 1 << b
        return dict(kind=kind, n=n, fs=2048.0, f_low=5.0 if low else 20.0, dtype="f32",
                    refs=min(_log_int(rng, 1, 24), max(1, (6 << 23) >> b)), W=_log_int(rng, n // 16, n))
    if kind == "mf_ref":
        f64 = rng.random() < 0.4
        n = 1 << (rng.randint(13, 17) if f64 else rng.randint(14, 21))
        return dict(kind=kind, n=n, fs=1024.0 if f64 else 2048.0, f_low=40.0 if f64 else 20.0,
                    dtype="f64" if f64 else "f32", refs=rng.randint(1, 3), pn=rng.choice([2, 7]))
    if kind == "build":
        n = 1 << rng.randint(15, 19)
        return dict(kind=kind, n=n, fs=2048.0, f_low=20.0, dtype=rng.choice(["f32", "f64"]), k=_log_int(rng, 3, 48),
                    pn=7, spread=0.01 * min(1.0, n / 2.0 ** 18), n_build=rng.choice([0, 0, -1]),
                    real=rng.random() < 0.3)
    form = rng.choice(["short64", "tensor", "series", "peaks", "peaks", "long"])
    c = dict(kind=kind, fs=2048.0, f_low=20.0, dtype="f32", refs=1, algo="auto", prec="native",
             real=rng.random() < 0.3, layout="")
    if form in ("short64", "tensor"):
        n = 1 << rng.randint(13, 16)
        c.update(n=n, fs=1024.0, f_low=40.0, k=rng.randint(3, 16), tau0=0.002, tau1=rng.uniform(0.02, 0.08),
                 W=rng.choice([1024, 1000, 512]))
        c.update(dict(dtype="f64") if form == "short64" else dict(algo="gemm", prec=rng.choice(["bf16x6", "bf16x9"])))
    elif form == "series":
        b = rng.randint(15, 19)
        c.update(n=1 << b, k=min(_log_int(rng, 3, 64), (64 << 18) >> b), tau0=0.05,
                 tau1=min(3.0, (1 << b) / 2048.0 / 16), W=0, layout=rng.choice(["", TWO]))
    elif form == "peaks":
        n = 1 << rng.randint(17, 20)
        c.update(n=n, refs=rng.randint(1, 4), k=_log_int(rng, 8, 64), tau0=0.05, tau1=n / 2048.0 / 35,
                 W=_log_int(rng, n // 8, n), layout=rng.choice(["", TWO, TWO]))
    else:
        n = 1 << rng.randint(21, 23)
        c.update(n=n, f_low=5.0, refs=rng.randint(1, 2), k=_log_int(rng, 12, 48), tau0=0.05,
                 tau1=120.0 * n / 2.0 ** 23, W=_log_int(rng, n // 8, n), layout=THREE, real=False)
    return c


# ------------------------------------------------------------------------------- inputs
def _dev():
    return "cuda"


def _gen(seed, stream):
    g = torch.Generator(device=_dev())
    g.manual_seed(1000 * int(seed) + stream)
    return g


def _freqs(case, n=None):
    n = n or case["n"]
    return torch.arange(n // 2 + 1, dtype=torch.float64, device=_dev()) * (case["fs"] / n)


def _inv_psd(f):
    """1 / S_n of an aLIGO-like fit (x = f / 215 Hz), 0 at DC."""
    x = torch.clamp(f, min=1e-3) / 215.0
    s = x ** -4.14 - 5.0 / x ** 2 + 111.0 * (1.0 - x ** 2 + 0.5 * x ** 4) / (1.0 + 0.5 * x ** 2)
    return torch.where(f > 0, 1.0 / s, torch.zeros_like(s))


def _f_high(case):
    return case["fs"] / 2 - DF_HIGH


def _band(case, f):
    return (f >= case["f_low"]) & (f <= _f_high(case))


def _strain(case, seed):
    """Coloured noise from f_low / 2 up, real[n] of the grid's type."""
    f = _freqs(case)
    w = torch.randn((2, f.numel()), dtype=torch.float64, device=_dev(), generator=_gen(seed, 0))
    ip = _inv_psd(f)
    amp = torch.where((f >= case["f_low"] / 2) & (ip > 0), 1.0 / torch.sqrt(torch.clamp(ip, min=1e-300)),
                      torch.zeros_like(f)) * math.sqrt(case["n"] / case["fs"] / 4.0)
    x = torch.fft.irfft(torch.complex(w[0] * amp, w[1] * amp), n=case["n"]) * case["fs"]
    return x.to(torch.float64 if case["dtype"] == "f64" else torch.float32)


class Template:
    """Component masses in M_sun, coalescence at time 0 and phase 0."""

    def __init__(self, m1, m2):
        self.m1, self.m2, self.tc, self.phic = float(m1), float(m2), 0.0, 0.0

    @staticmethod
    def of(mchirp, eta):
        m = mchirp / eta ** 0.6
        d = math.sqrt(max(0.0, 1.0 - 4.0 * eta))
        return Template(0.5 * m * (1.0 + d), 0.5 * m * (1.0 - d))


def _references(case, seed):
    r = np.random.default_rng([int(seed), 7])
    return [Template.of(r.uniform(1.0, 2.4), r.uniform(0.24, 0.25)) for _ in range(case["refs"])]


def _newton_phase(case, mchirp, f):
    """Leading-order stationary phase of a chirp mass (M_sun)."""
    return 3.0 / 128.0 * (math.pi * MSUN_S * mchirp * torch.clamp(f, min=1e-3)) ** (-5.0 / 3.0)


def _filters(case, seed):
    """Stored filters (4 / (n N)) conj(h~) / S_n on the band, [refs, n/2+1]."""
    f = _freqs(case)
    ip, band = _inv_psd(f), _band(case, f)
    b = torch.where(band, torch.clamp(f, min=1e-3) ** (-7.0 / 6.0), torch.zeros_like(f))
    norm = torch.sqrt(4.0 * case["fs"] / case["n"] * torch.sum(b * b * ip))
    ct = torch.complex128 if case["dtype"] == "f64" else torch.complex64
    out = torch.empty((case["refs"], f.numel()), dtype=ct, device=_dev())
    for r, t in enumerate(_references(case, seed)):
        mc = (t.m1 * t.m2) ** 0.6 / (t.m1 + t.m2) ** 0.2
        out[r] = torch.polar(4.0 / (case["n"] * norm) * b * ip, _newton_phase(case, mc, f)).to(ct)
    return out


def _series(case, seed):
    """Reference SNR series [refs, n]: band-limited analytic noise with unit variance per part."""
    f = _freqs(case)
    g = _gen(seed, 1)
    amp = torch.where(_band(case, f), torch.sqrt(_inv_psd(f)) * torch.clamp(f, min=1e-3) ** (-7.0 / 6.0),
                      torch.zeros_like(f))
    amp = amp * math.sqrt(2.0) / torch.sqrt(torch.sum(amp * amp))
    ct = torch.complex128 if case["dtype"] == "f64" else torch.complex64
    z = torch.empty((case["refs"], case["n"]), dtype=ct, device=_dev())
    for r in range(case["refs"]):
        w = torch.randn((2, f.numel()), dtype=torch.float64, device=_dev(), generator=g)
        full = torch.zeros(case["n"], dtype=torch.complex128, device=_dev())
        full[: f.numel()] = torch.complex(w[0] * amp, w[1] * amp) * (case["n"] / math.sqrt(2.0))
        z[r] = torch.fft.ifft(full).to(ct)
    return z


def _window(case, f, dfl):
    """Cosine tapers of dfl below f_low and DF_HIGH above f_high."""
    lo, hi = case["f_low"], _f_high(case)
    w = torch.where((f >= lo) & (f <= hi), torch.ones_like(f), torch.zeros_like(f))
    w = torch.where((f > lo - dfl) & (f < lo), 0.5 * (1.0 + torch.cos(math.pi * (f - lo) / dfl)), w)
    return torch.where((f > hi) & (f < hi + DF_HIGH),
                       0.5 * (1.0 - torch.cos(math.pi * (f - (hi + DF_HIGH)) / DF_HIGH)), w)


def _kernels(case, seed):
    """Per reference: (lag0, length, packed host taps of the grid's type) of k neighbours whose
    time offset at f_low is spread over tau0 .. tau1 seconds, both signs."""
    r = np.random.default_rng([int(seed), 3])
    dfl = min(DF_LOW_MAX, 0.5 * case["f_low"])
    out = []
    for _ in range(case["refs"]):
        lag0, length, taps = [], [], []
        for j in range(case["k"]):
            u = (j // 2 + r.uniform(0.0, 1.0)) / max(1, (case["k"] + 1) // 2)
            tau = case["tau0"] * (case["tau1"] / case["tau0"]) ** min(1.0, u) * (1.0 if j % 2 else -1.0)
            nb = 1 << 12
            while nb < min(case["n"], 4 * case["fs"] * (abs(tau) * 2.5 + 4.0 / dfl)):
                nb *= 2
            f = _freqs(case, nb)
            ph = 2.0 * math.pi * 0.6 * tau * case["f_low"] * (torch.clamp(f, min=1e-3) / case["f_low"]) ** (-5.0 / 3.0)
            full = torch.zeros(nb, dtype=torch.complex128, device=_dev())
            full[: f.numel()] = torch.polar(_window(case, f, dfl), ph)
            rho = torch.fft.ifft(full)
            if case["real"]:
                rho = torch.complex(2.0 * rho.real, torch.zeros_like(rho.real))
            rho = torch.fft.fftshift(rho)
            mag = rho.abs()
            kept = torch.nonzero(mag >= THRESHOLD * mag.max())
            a, b = int(kept[0]), int(kept[-1]) + 1
            lag0.append(a - nb // 2)
            length.append(b - a)
            taps.append(rho[a:b])
        t = torch.cat(taps)
        f64 = case["dtype"] == "f64"
        if case["real"]:
            t = t.real.to(torch.float64 if f64 else torch.float32)
        else:
            t = t.to(torch.complex128 if f64 else torch.complex64)
        out.append((np.array(lag0, np.int32), np.array(length, np.int32), t.cpu().numpy()))
    return out


def _bank(case, seed):
    """A reference and k neighbours within `spread` of its chirp mass."""
    r = np.random.default_rng([int(seed), 5])
    mc = r.uniform(1.2, 1.6)
    ref = Template.of(mc, 0.2495)
    nbrs = [Template.of(mc * (1.0 + case["spread"] * r.uniform(-1.0, 1.0)), r.uniform(0.235, 0.25))
            for _ in range(case["k"])]
    return ref, nbrs


def _store(case):
    """The store that the packed taps of the set go to, with room for the longest kernels."""
    rt, ct = (torch.float64, torch.complex128) if case["dtype"] == "f64" else (torch.float32, torch.complex64)
    return torch.zeros(case["k"] * min(case["n"], 1 << 15), dtype=rt if case["real"] else ct, device=_dev())


def _put(store, taps):
    store[: taps.numel()] = taps
    return store


def _context(case):
    return RatioFilter(case["n"], case["fs"], case["f_low"], _f_high(case), case.get("pn", 7), case["dtype"],
                       DF_HIGH, DF_LOW_MAX)


def prepare(case, seed):
    s = dict(case=case, rf=_context(case))
    if case["kind"] == "mf":
        s.update(x=_strain(case, seed), filt=_filters(case, seed))
    elif case["kind"] == "mf_ref":
        s.update(x=_strain(case, seed), inv_psd=_inv_psd(_freqs(case)), refs=_references(case, seed))
    elif case["kind"] == "build":
        ref, nbrs = _bank(case, seed)
        s.update(inv_psd=_inv_psd(_freqs(case)), ref=ref, nbrs=nbrs, store=_store(case))
    else:
        z = _series(case, seed)
        kern = [s["rf"].kernels_import(*kt, real=case["real"]) for kt in _kernels(case, seed)]
        if case["layout"]:
            spec = [b.split(":") for b in case["layout"].split(",")]
            for k in kern:
                k.prepare_forms([int(b[0]) for b in spec], [b[3] if len(b) > 3 else "os" for b in spec],
                                ["native"] * len(spec), [int(b[1]) for b in spec], [int(b[2]) for b in spec])
        s.update(z=[z[g] for g in range(case["refs"])], kern=kern)
    return s


def run(s):
    case, rf = s["case"], s["rf"]
    if case["kind"] == "mf":
        z = rf.mf_filtered(s["x"], s["filt"])
        if not case["W"]:
            return dict(z=z)
        peak, arg = rf.winmax(z, case["W"])
        return dict(z=z, peak=peak, arg=arg)
    if case["kind"] == "mf_ref":
        z, sigma = rf.mf_reference(s["x"], s["inv_psd"], s["refs"])
        return dict(z=z, sigma=sigma)
    if case["kind"] == "build":
        k = rf.build_ratio_kernels(s["ref"], s["nbrs"], s["inv_psd"], THRESHOLD, n_build=case["n_build"],
                                   real=case["real"])
        return dict(taps=_put(s["store"], k.taps()), lag0=k.lag0, length=k.length)
    if not case["W"]:
        return dict(z=rf.reconstruct(s["z"][0], s["kern"][0], case["algo"], prec=case["prec"]))
    if case["refs"] == 1:
        peak, arg = rf.reconstruct_winmax(s["z"][0], s["kern"][0], case["W"], case["algo"], prec=case["prec"])
    else:
        peak, arg = rf.reconstruct_batched(s["z"], s["kern"], case["W"], case["algo"], prec=case["prec"])
    return dict(peak=peak, arg=arg)


def work(case):
    """Bytes: the inputs read and the outputs written once.  Operations: a transform of the data
    and of each series (5 n log2 n), or for a reconstruction the cheaper of the direct sum and
    one block transform per output of blocks of twice the typical kernel plus one product."""
    n, r = case["n"], 8 if case["dtype"] == "f64" else 4
    fft = 5.0 * n * math.log2(n)
    nw = -(-n // case["W"]) if case.get("W") else 0
    if case["kind"] == "mf":
        return {"bytes": n * r + case["refs"] * (n * r + 2 * n * r + 8 * nw), "flops": fft / 2 + case["refs"] * (fft + 5 * n)}
    if case["kind"] == "mf_ref":
        return {"bytes": n * r + 4 * n + case["refs"] * 2 * n * r, "flops": fft / 2 + case["refs"] * (fft + 15 * n)}
    length = 0.4 * case["fs"] if case["kind"] == "build" else \
        case["fs"] * (math.sqrt(case["tau0"] * case["tau1"]) + 4.0 / min(DF_LOW_MAX, 0.5 * case["f_low"]))
    if case["kind"] == "build":
        return {"bytes": 4 * n + case["k"] * length * 2 * r, "flops": case["k"] * (fft + 20 * n)}
    rows = case["refs"] * case["k"]
    per = min((4.0 if case["real"] else 8.0) * length, 10.0 * math.log2(2.0 * length) + 8.0)
    out = rows * (8 * nw if case["W"] else 2 * r * n)
    return {"bytes": case["refs"] * 2 * r * n + rows * length * r * (1 if case["real"] else 2) + out,
            "flops": rows * n * per}


# ------------------------------------------------------------------------------- 64-bit results
def _peaks(case, z):
    """Window peaks of one series: (max |z|^2 as float64, first index)."""
    n, W = case["n"], case["W"]
    m = z.real ** 2 + z.imag ** 2
    nw = -(-n // W)
    m = torch.nn.functional.pad(m, (0, nw * W - n), value=-1.0).reshape(nw, W)
    v, i = torch.max(m, dim=1)
    return v, (i + torch.arange(nw, device=_dev()) * W).to(torch.int32)


def _tf2_phase(t, f, pn):
    """Non-spinning TaylorF2 phase (Buonanno, Iyer, Ochsner, Pan & Sathyaprakash 2009)."""
    m, pi = t.m1 + t.m2, math.pi
    e = t.m1 * t.m2 / (m * m)
    v = (pi * m * MSUN_S * torch.clamp(f, min=1e-6)) ** (1.0 / 3.0)
    g = torch.ones_like(v)
    if pn >= 2:
        g = g + (3715.0 / 756.0 + 55.0 / 9.0 * e) * v ** 2
    if pn >= 3:
        g = g - 16.0 * pi * v ** 3
    if pn >= 4:
        g = g + (15293365.0 / 508032.0 + 27145.0 / 504.0 * e + 3085.0 / 72.0 * e * e) * v ** 4
    if pn >= 5:
        g = g + pi * (38645.0 / 756.0 - 65.0 / 9.0 * e) * (1.0 + 3.0 * torch.log(v * math.sqrt(6.0))) * v ** 5
    if pn >= 6:
        a6 = (11583231236531.0 / 4694215680.0 - 640.0 / 3.0 * pi * pi - 6848.0 / 21.0 * 0.57721566490153286061 +
              (-15737765635.0 / 3048192.0 + 2255.0 / 12.0 * pi * pi) * e + 76055.0 / 1728.0 * e * e -
              127825.0 / 1296.0 * e ** 3)
        g = g + (a6 - 6848.0 / 21.0 * torch.log(4.0 * v)) * v ** 6
    if pn >= 7:
        g = g + pi * (77096675.0 / 254016.0 + 378515.0 / 1512.0 * e - 74045.0 / 756.0 * e * e) * v ** 7
    return -0.25 * pi + 3.0 / (128.0 * e) * g * v ** -5.0


def _tf2_tau_slope(t, f0, pn):
    """d/df of Psi' / (2 pi) at f0 (1/Hz^2 s), by differentiation of the phase."""
    f = torch.tensor([f0], dtype=torch.float64, device=_dev(), requires_grad=True)
    d1 = torch.autograd.grad(_tf2_phase(t, f, pn).sum(), f, create_graph=True)[0]
    return float(torch.autograd.grad(d1.sum(), f)[0]) / (2.0 * math.pi)


def exact(case, seed):
    n = case["n"]
    if case["kind"] in ("mf", "mf_ref"):
        f = _freqs(case)
        X = torch.fft.rfft(_strain(case, seed).to(torch.float64))
        if case["kind"] == "mf":
            filt, sigma = _filters(case, seed), None
        else:
            ip, band = _inv_psd(f), _band(case, f)
            b = torch.where(band, torch.clamp(f, min=1e-3) ** (-7.0 / 6.0), torch.zeros_like(f))
            sg = torch.sqrt(4.0 * case["fs"] / n * torch.sum(b * b * ip))
            refs = _references(case, seed)
            sigma = sg.repeat(len(refs))
        z = torch.empty((case["refs"], n), dtype=torch.complex128, device=_dev())
        for r in range(case["refs"]):
            F = filt[r].to(torch.complex128) if sigma is None else \
                torch.polar(4.0 / (n * sg) * b * ip, _tf2_phase(refs[r], f, case["pn"]))
            full = torch.zeros(n, dtype=torch.complex128, device=_dev())
            full[: n // 2 + 1] = X * F
            z[r] = torch.fft.ifft(full) * n
        if sigma is not None:
            return dict(z=z, sigma=sigma)
        if not case["W"]:
            return dict(z=z)
        p = [_peaks(case, z[r]) for r in range(case["refs"])]
        return dict(z=z, peak=torch.stack([v for v, _ in p]), arg=torch.stack([i for _, i in p]))
    if case["kind"] == "build":
        if case["n_build"]:
            return None   # a grid per neighbour, by a rule of the library's own
        ref, nbrs = _bank(case, seed)
        f = _freqs(case)
        pr = _tf2_phase(ref, f, case["pn"])
        sr = _tf2_tau_slope(ref, case["f_low"], case["pn"])
        taps, lag0, length = [], [], []
        for t in nbrs:
            ds = abs(_tf2_tau_slope(t, case["f_low"], case["pn"]) - sr)
            dfl = min(DF_LOW_MAX, 0.5 * case["f_low"], 1.0 / math.sqrt(ds) if ds > 0 else math.inf)
            full = torch.zeros(n, dtype=torch.complex128, device=_dev())
            full[: n // 2 + 1] = torch.polar(_window(case, f, dfl), _tf2_phase(t, f, case["pn"]) - pr)
            full[0] = 0
            rho = torch.fft.ifft(full)
            if case["real"]:
                rho = torch.complex(2.0 * rho.real, torch.zeros_like(rho.real))
            mag = rho.real ** 2 + rho.imag ** 2
            kept = torch.nonzero(mag >= THRESHOLD * THRESHOLD * mag.max()).flatten()
            gap = torch.cat([kept[1:] - kept[:-1], kept[:1] + n - kept[-1:]])
            at = int(torch.argmax(gap))
            m0, m1 = int(kept[(at + 1) % kept.numel()]), int(kept[at])
            L = (m1 - m0) % n + 1
            c = rho[(m0 + torch.arange(L, device=_dev())) % n]
            taps.append(c.real if case["real"] else c)
            lag0.append(m0 if m0 <= n // 2 else m0 - n)
            length.append(L)
        return dict(taps=_put(_store(case).to(taps[0].dtype), torch.cat(taps)), lag0=np.array(lag0, np.int64), length=np.array(length, np.int64))
    zs = _series(case, seed)
    rows = []
    for g, (lag0, length, taps) in enumerate(_kernels(case, seed)):
        Z = torch.fft.fft(zs[g].to(torch.complex128))
        t = torch.from_numpy(taps).to(_dev()).to(torch.complex128)
        o = 0
        for j in range(case["k"]):
            L = int(length[j])
            c = torch.zeros(n, dtype=torch.complex128, device=_dev())
            c[(int(lag0[j]) + torch.arange(L, device=_dev())) % n] = t[o:o + L]
            o += L
            z = torch.fft.ifft(Z * torch.fft.fft(c))
            rows.append(_peaks(case, z) if case["W"] else z)
    if not case["W"]:
        return dict(z=torch.stack(rows))
    return dict(peak=torch.stack([v for v, _ in rows]), arg=torch.stack([i for _, i in rows]))
