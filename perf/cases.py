"""What is timed: the calls that a search built on this library makes.

Every case goes through the binding (``mf.Plan``, ``mf.Batch``, ``mf.MLP``,
``mf.psd_welch``, ``Hierarchy``), on synthetic two-detector data: coloured
Gaussian noise of the analytic PSD, TaylorF2 signals of the case's own bank and
sine-Gaussian glitches.  Kinds:

``segment``   strain -> spectrum -> filter -> triggers on the host.
``filter``    spectra -> filter -> triggers on the host, with the storage of the
              bank, of the data and of the intermediate as options.
``stage1``    the coarse stage: filter, time-shifted coincidences, follow-up flags.
``veto``      chi^2 and sine-Gaussian chi^2 at the triggers of a filter run.
``hierarchy`` the whole two-stage step from host strain.
``batch``     long data against length classes of templates.
``psd``       Welch estimate of the data's PSD.
``bank``      templates generated into a plan's bank, with their norms.
``proposal``  the ranking network: a training step, or the ranked slots.
"""

from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2309_00019_gb300 import mf
from paper_2309_00019_gb300.hierarchy import Hierarchy, HierParams

DEV = "cuda:0"
MTSUN = 4.925491025543576e-06
DTYPE = {"f32": mf.MF_F32, "f16": mf.MF_F16, "bf16": mf.MF_BF16, "f16x2": mf.MF_F16X2}
CLASS_LEN = (4.0, 16.0, 64.0, 256.0)


# -- the cases ------------------------------------------------------------------

def listed():
    return [
        # One 32 s segment of one detector at 512 Hz against a handful of templates: the smallest search
        # there is, where launches, copies and waits are what a user waits for.
        dict(name="segment 16k", kind="segment", lg=14, fs=512.0, dets=1, tmpl=64, thr=5.5, window=512),
        # A short segment at 4096 Hz with a bfloat16 bank and bfloat16 data, a ragged clustering window and an
        # odd number of selected templates: the reduced-precision path on ordinary sizes.
        dict(name="filter bf16 128k", kind="filter", lg=17, fs=4096.0, dets=2, tmpl=600, sel=501, thr=5.5,
             window=3000, bank="bf16", data="bf16", inter="f32"),
        # The coarse stage of the two-stage search at its full size: 2,000 templates on 512 s at 512 Hz.
        dict(name="stage 1 256k", kind="stage1", lg=18, fs=512.0, dets=2, tmpl=2000, thr=3.5, window=512,
             shift=2560, shifts=101, rho_c=7.0),
        # The fine stage as the search runs it: a selection of the fine bank on 512 s at 2048 Hz with the FP16
        # intermediate.  Most of the search's time goes here.
        dict(name="stage 2 1M f16", kind="filter", lg=20, fs=2048.0, dets=2, tmpl=1400, sel=1031, thr=4.0,
             window=2048, bank="f32", data="f32", inter="f16"),
        # The same call with the library's defaults, everything in FP32.
        dict(name="filter 1M f32", kind="filter", lg=20, fs=2048.0, dets=2, tmpl=320, sel=-1, thr=5.5,
             window=2048, bank="f32", data="f32", inter="f32"),
        # The reduced-precision workload: FP16 bank and FP16 data on 256 s at 4096 Hz.
        dict(name="filter 1M f16 bank", kind="filter", lg=20, fs=4096.0, dets=2, tmpl=400, sel=-1, thr=5.5,
             window=4096, bank="f16", data="f16", inter="f32"),
        # Long data in overlapping segments against templates of uneven length, as one fused queue.
        dict(name="batch uneven", kind="batch", lg=20, fs=2048.0, dets=2, secs=1024, per="20,210,150,20",
             thr=5.5, inter="f16"),
        # The whole two-stage step from host strain to triggers and coincidences on the host.
        dict(name="hierarchy", kind="hierarchy", lg=20, coarse=400, fine=2400, near=40, thr=3.5, thr2=4.0,
             rho_c=7.0, inter="f16"),
        # The vetoes at the triggers of a stage-2 run.
        dict(name="veto 256k", kind="veto", lg=18, fs=2048.0, dets=2, tmpl=150, thr=4.5, window=2048, bands=16,
             bank="f32"),
        # The PSD of the data that are analysed, before the filter.
        dict(name="psd median", kind="psd", lg=14, fs=2048.0, dets=2, samples=1 << 20, stride=8192,
             average="median"),
        # Templates into the bank: done once per search, over thousands of templates, and the start of each run.
        dict(name="bank 1M", kind="bank", lg=20, fs=2048.0, tmpl=384, bank="f32"),
        # One training step of the ranking network at its own sizes.
        dict(name="proposal step", kind="proposal", train=True, batch=1024, width=256, depth=4, slots=2000, k=16),
    ]


def draw(rng):
    def near(a, b):  # spread over the logarithm, odd values among them
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["segment", "filter", "filter", "filter", "filter", "stage1", "veto", "hierarchy", "batch", "psd",
                       "bank", "proposal"])
    fs = rng.choice([512.0, 1024.0, 2048.0, 4096.0])
    if kind == "segment":
        lg = rng.randint(12, 17)
        return dict(kind=kind, lg=lg, fs=fs, dets=rng.randint(1, 3), tmpl=near(1, 400), thr=5.5,
                    window=rng.choice([int(fs), near(100, 1 << lg)]))
    if kind == "filter":
        lg = rng.choice([13, 14, 15, 16, 17, 18, 19, 20, 20, 20])
        top = min(3000, 700 << (20 - lg))
        bank = rng.choice(["f32", "f32", "f32", "f16", "bf16"])
        inter = rng.choice(["f32", "f16", "f16", "f16x2"]) if lg == 20 else "f32"
        data = rng.choice(["f32", bank]) if inter == "f32" else "f32"
        tmpl = near(8, top)
        return dict(kind=kind, lg=lg, fs=fs, dets=rng.choice([1, 2, 2, 2, 3]), tmpl=tmpl,
                    sel=rng.choice([-1, rng.randint(1, tmpl)]), thr=rng.choice([4.0, 4.5, 5.5]),
                    window=rng.choice([int(fs), near(500, 1 << lg)]), bank=bank, data=data, inter=inter)
    if kind == "stage1":
        lg = rng.randint(14, 18)
        return dict(kind=kind, lg=lg, fs=512.0, dets=2, tmpl=near(30, 2000), thr=rng.choice([3.5, 4.0]), window=512,
                    shift=rng.choice([2560, near(300, 2000)]), shifts=near(3, 101), rho_c=rng.choice([6.5, 7.0]))
    if kind == "veto":
        lg = rng.randint(14, 18)
        return dict(kind=kind, lg=lg, fs=fs, dets=rng.randint(1, 2), tmpl=near(10, 150), thr=rng.choice([4.5, 5.0]),
                    window=int(fs), bands=rng.choice([8, 13, 16]), bank=rng.choice(["f32", "f32", "f16"]))
    if kind == "hierarchy":
        lg = rng.randint(16, 20)
        return dict(kind=kind, lg=lg, coarse=near(40, 400), fine=near(200, 2400), near=near(5, 40), thr=3.5, thr2=4.0,
                    rho_c=7.0, inter="f32" if lg < 20 else rng.choice(["f16", "f32"]))
    if kind == "batch":
        lg = rng.choice([18, 19, 20, 20])
        per = [near(4, 20), near(20, 180), near(20, 120), 0 if lg < 20 else near(2, 20)]
        return dict(kind=kind, lg=lg, fs=2048.0, dets=rng.randint(1, 2), secs=rng.randint(300, 1024), per=",".join(map(str, per)),
                    thr=5.5, inter="f32" if lg < 20 else rng.choice(["f16", "f32"]))
    if kind == "psd":
        lg = rng.randint(12, 16)
        return dict(kind=kind, lg=lg, fs=fs, dets=rng.randint(1, 2), samples=near(4 << lg, 1 << 20),
                    stride=rng.choice([1 << lg, 1 << (lg - 1), rng.randint(1 << (lg - 2), 1 << lg)]),
                    average=rng.choice(["median", "mean"]))
    if kind == "bank":
        lg = rng.randint(14, 20)
        return dict(kind=kind, lg=lg, fs=fs, tmpl=near(8, min(2000, 360 << (20 - lg))), bank=rng.choice(["f32", "f32", "f16"]))
    return dict(kind="proposal", train=rng.random() < 0.5, batch=near(16, 1024), width=256, depth=4,
                slots=near(200, 2000), k=rng.randint(4, 32))


# -- inputs -----------------------------------------------------------------------

def psd_bins(n, fs):
    """The analytic one-sided PSD on bins 0..n/2 (0 at DC), host float64."""
    x = np.arange(n // 2 + 1, dtype=np.float64) * (fs / n) / 215.0
    with np.errstate(divide="ignore", invalid="ignore"):
        s = 1e-46 * (x ** -4.14 - 5.0 * x ** -2 + 111.0 * (1.0 - x ** 2 + 0.5 * x ** 4) / (1.0 + 0.5 * x ** 2))
    s[0] = 0.0
    return s


def masses(rng, count):
    """Component masses: chirp masses of 1.2 to 10, mass ratios of 0.2 to 1."""
    mc = np.exp(rng.uniform(math.log(1.2), math.log(10.0), count))
    q = rng.uniform(0.2, 1.0, count)
    m1 = mc * (1 + q) ** 0.2 / q ** 0.6
    return m1, m1 * q


def f_isco(m1, m2):
    return 1.0 / (6.0 ** 1.5 * math.pi * (np.asarray(m1) + np.asarray(m2)) * MTSUN)


def waveforms(n, fs, m1, m2, f_low):
    """Templates f^{-7/6} exp(-i Psi), 2PN phase, complex64 [count, n/2 + 1] on the GPU."""
    nb = n // 2 + 1
    f = torch.arange(nb, dtype=torch.float64, device=DEV) * (fs / n)
    f[0] = f[1]
    amp = f.pow(-7.0 / 6.0).float()
    out = torch.empty((len(m1), nb), dtype=torch.complex64, device=DEV)
    step = max(1, (1 << 25) // nb)
    cube = f.pow(1.0 / 3.0)
    for a in range(0, len(m1), step):
        p = torch.from_numpy(np.stack([m1[a:a + step], m2[a:a + step]])).to(DEV)
        mt = (p[0] + p[1])[:, None]
        eta = (p[0] * p[1])[:, None] / mt ** 2
        v = (math.pi * MTSUN * mt) ** (1.0 / 3.0) * cube[None, :]
        psi = 1 + v * v * ((3715.0 / 756 + 55.0 / 9 * eta) + v * (-16 * math.pi + v * (
            15293365.0 / 508032 + 27145.0 / 504 * eta + 3085.0 / 72 * eta * eta)))
        psi = 3.0 / (128.0 * eta) * psi / (v ** 5)
        psi = torch.remainder(psi, 2 * math.pi).float()
        fi = torch.from_numpy(np.minimum(f_isco(m1[a:a + step], m2[a:a + step]), fs / 2)).to(DEV)[:, None]
        keep = ((f[None, :] >= f_low) & (f[None, :] <= fi)).float() * amp[None, :]
        out[a:a + step] = torch.complex(keep * torch.cos(psi), -keep * torch.sin(psi))
    out[:, 0] = 0
    out[:, nb - 1] = 0
    return out


def weights(n, fs, f_low):
    """4 df / S_n on the band f_low <= f < fs / 2, float64 on the GPU."""
    s = torch.from_numpy(psd_bins(n, fs)).to(DEV)
    k = torch.arange(n // 2 + 1, device=DEV)
    band = (k >= math.ceil(f_low * n / fs - 1e-9)) & (k > 0) & (k < n // 2) & (s > 0)
    return torch.where(band, 4.0 * (fs / n) / torch.where(band, s, torch.ones_like(s)), torch.zeros_like(s))


def spectra(gen, rng, n, fs, dets, f_low, m1, m2, signals, glitches):
    """Noise, signals of the given masses at SNR 6 to 20 and glitches at SNR 8 to 50: complex128 [dets, n/2 + 1]."""
    nb, T = n // 2 + 1, n / fs
    f = torch.arange(nb, dtype=torch.float64, device=DEV) * (fs / n)
    s = torch.from_numpy(psd_bins(n, fs)).to(DEV)
    keep = (f >= 10.0) & (torch.arange(nb, device=DEV) < n // 2)
    sd = torch.where(keep, torch.sqrt(torch.clamp(T * s / 4.0, min=0.0)), torch.zeros_like(s))
    x = torch.randn((dets, nb, 2), dtype=torch.float64, device=DEV, generator=gen)
    d = sd * torch.view_as_complex(x)
    w = weights(n, fs, f_low)
    pick = rng.integers(0, len(m1), signals)
    t0 = (np.arange(signals) + rng.uniform(0.2, 0.8, signals)) * T / max(1, signals)
    for i in range(signals):
        h = waveforms(n, fs, m1[pick[i]:pick[i] + 1], m2[pick[i]:pick[i] + 1], f_low)[0].to(torch.complex128)
        h = h * (rng.uniform(6.0, 20.0) / torch.sqrt((w * (h.real ** 2 + h.imag ** 2)).sum()))
        for j in range(dets):
            t = t0[i] + (rng.uniform(-0.01, 0.01) if j else 0.0)
            d[j] += h * torch.polar(torch.ones_like(f), torch.remainder(-2 * math.pi * f * t + rng.uniform(0, 6.28), 2 * math.pi))
    for j in range(dets):
        for _ in range(glitches):
            f0, q, t = rng.uniform(f_low, min(500.0, 0.4 * fs)), rng.uniform(5.0, 20.0), rng.uniform(0.02, 0.98) * T
            g = torch.exp(-(math.pi * q / (math.sqrt(2.0) * math.pi * f0) * (f - f0)) ** 2)
            g = g * (rng.uniform(8.0, 50.0) / torch.sqrt((w * g * g).sum()))
            d[j] += g * torch.polar(torch.ones_like(f), torch.remainder(-2 * math.pi * f * t, 2 * math.pi))
    d[:, 0] = 0
    d[:, nb - 1] = 0
    return d


def noise_strain(gen, rng, n, fs, dets, count, f_low, m1, m2, signals, glitches):
    """The first `count` samples of n, float32 [dets, count] on the GPU."""
    d = spectra(gen, rng, n, fs, dets, f_low, m1, m2, signals, glitches)
    return (torch.fft.irfft(d, n=n, dim=-1) * fs)[:, :count].to(torch.float32).contiguous()


def rngs(seed):
    return np.random.default_rng(seed), torch.Generator(device=DEV).manual_seed(seed)


def low_cut(fs):
    return 30.0


# -- states ------------------------------------------------------------------------

def put_bank(plan, n, fs, m1, m2, f_low, dtype):
    """A user's templates into the plan's bank in blocks of rows."""
    plan.bank_reserve(len(m1), dtype)
    step = max(1, (1 << 26) // (n // 2 + 1))
    for a in range(0, len(m1), step):
        rows = waveforms(n, fs, m1[a:a + step], m2[a:a + step], f_low)
        if dtype == mf.MF_F32:
            plan.bank_set_rows(a, rows)
        else:
            plan.bank_quantize_rows(a, rows)


def search_inputs(c, seed):
    """(m1, m2, spectra complex64, selection) of the kinds that filter one segment."""
    rng, gen = rngs(seed)
    n, fs = 1 << c["lg"], c["fs"]
    m1, m2 = masses(rng, c["tmpl"])
    T = n / fs
    d = spectra(gen, rng, n, fs, c["dets"], low_cut(fs), m1, m2, max(1, int(T / 16)), max(1, int(T / 32)))
    sel = None
    if c.get("sel", -1) >= 0:
        sel = np.sort(rng.choice(c["tmpl"], c["sel"], replace=False)).astype(np.int32)
    return m1, m2, d.to(torch.complex64).contiguous(), sel


def search_plan(c, m1, m2):
    n, fs = 1 << c["lg"], c["fs"]
    p = mf.Plan(fs, n, c["dets"], low_cut(fs), fs / 2, c["thr"], c["window"], dtype=DTYPE[c.get("bank", "f32")],
                max_triggers=1 << 22)
    p.set_psd(psd_bins(n, fs))
    put_bank(p, n, fs, m1, m2, low_cut(fs), DTYPE[c.get("bank", "f32")])
    if c.get("data", "f32") != "f32":
        p.set_data_dtype(DTYPE[c["data"]])
    if c.get("inter", "f32") != "f32":
        p.set_intermediate(DTYPE[c["inter"]])
    return p


def prepare(case, seed):
    c, kind = case, case["kind"]
    rng, gen = rngs(seed + 7)
    if kind in ("segment", "filter", "stage1", "veto"):
        m1, m2, d, sel = search_inputs(c, seed)
        n, fs = 1 << c["lg"], c["fs"]
        s = dict(kind=kind, c=c, plan=search_plan(c, m1, m2), d=d)
        s["sel"] = None if sel is None else torch.from_numpy(sel).to(DEV)
        wins = (c["sel"] if sel is not None else c["tmpl"]) * c["dets"] * -(-n // c["window"])
        s["cap"] = capacity(wins, c["thr"])
        if kind in ("segment", "filter"):
            s["rec"] = records(mf.TRIGGER_NP, s["cap"])
        if kind == "segment":
            s["strain"] = (torch.fft.irfft(d.to(torch.complex128), n=n, dim=-1) * fs).to(torch.float32).contiguous()
            s["d"] = torch.zeros_like(d)
        if kind == "stage1":
            s["rec"] = records(mf.COINC_NP, 1 << 17)
            s["followed"] = torch.zeros(c["tmpl"], dtype=torch.int32, device=DEV)
        if kind == "veto":  # the triggers are there: the vetoes follow the filter that found them
            s["plan"].filter(d)
            s["out"] = [torch.zeros(1 << 22, device=DEV) for _ in range(4)]
            s["f_final"] = torch.from_numpy(f_isco(m1, m2)).to(DEV, torch.float32)
            s["mtotal"] = torch.from_numpy(m1 + m2).to(DEV, torch.float32)
        return s
    if kind == "hierarchy":
        n2, fs2 = 1 << c["lg"], 2048.0
        n1, fs1 = n2 // 4, 512.0
        cm, fm = masses(rng, c["coarse"]), masses(rng, c["fine"])
        # neighbourhood of a coarse template: the fine templates nearest to it in chirp mass and mass ratio
        place = lambda m: np.stack([15 * np.log((m[0] * m[1]) ** 0.6 / (m[0] + m[1]) ** 0.2), m[1] / m[0]])  # noqa: E731
        a, b = place(cm), place(fm)
        dist = ((a[:, :, None] - b[:, None, :]) ** 2).sum(axis=0)
        idx = np.argsort(dist, axis=1, kind="stable")[:, :c["near"]].astype(np.int32)
        ptr = np.arange(c["coarse"] + 1, dtype=np.int64) * idx.shape[1]
        hp = HierParams(n2=n2, fs2=fs2, n1=n1, fs1=fs1, f_low=30.0, thr1=c["thr"], thr2=c["thr2"], window1=512,
                        window2=2048, shift_s=5.0 if n2 >= 1 << 20 else 2.0, n_shifts=101 if n2 >= 1 << 20 else 5,
                        coinc_s=0.015, rho_c_thr=c["rho_c"], max_trig1=1 << 20, max_trig2=1 << 23)
        h = Hierarchy(hp, psd_bins(n1, fs1), psd_bins(n2, fs2), c["coarse"], c["fine"], ptr, idx.reshape(-1))
        for stage, n, fs, m in ((1, n1, fs1, cm), (2, n2, fs2, fm)):
            step = max(1, (1 << 26) // (n // 2 + 1))
            for r in range(0, len(m[0]), step):
                h.set_bank_rows(stage, r, waveforms(n, fs, m[0][r:r + step], m[1][r:r + step], 30.0))
        if c["inter"] != "f32":
            h.p2.set_intermediate(DTYPE[c["inter"]])
        T = n2 / fs2
        x = noise_strain(gen, rng, n2, fs2, 2, n2, 30.0, *fm, max(2, int(T / 12)), max(1, int(T / 26)))
        return dict(kind=kind, c=c, h=h, strain=x.cpu().pin_memory(), co=records(mf.COINC_NP, 1 << 17),
                    rec=records(mf.TRIGGER_NP, capacity(c["fine"] * 2 * T, c["thr2"])))
    if kind == "batch":
        n, fs, count = 1 << c["lg"], c["fs"], int(c["secs"] * c["fs"])
        per = [int(v) for v in c["per"].split(",")]
        ls = CLASS_LEN[:len(per) if per[-1] else len(per) - 1]
        b = mf.Batch(fs, c["dets"], count, 25.0, fs / 2, c["thr"], int(fs), ls, max_triggers=1 << 20)
        b.set_psd(psd_bins(1 << 20, fs), 1 << 20)
        ms = []
        for i in range(len(ls)):
            b.set_segment(i, n)
            m = masses(rng, per[i])
            ms.append(m)
            p = b.plan(i)
            put_bank(p, n, fs, m[0], m[1], 25.0, mf.MF_F32)
            if c["inter"] != "f32":
                p.set_intermediate(DTYPE[c["inter"]])
        m = np.concatenate([np.stack(v) for v in ms], axis=1)
        x = noise_strain(gen, rng, 1 << (count - 1).bit_length(), fs, c["dets"], count, 25.0, m[0], m[1],
                         max(2, c["secs"] // 32), max(1, c["secs"] // 64))
        torch.cuda.synchronize()
        return dict(kind=kind, c=c, b=b, strain=x,
                    rec=records(mf.BATCH_TRIGGER_NP, capacity(sum(per) * c["dets"] * c["secs"], c["thr"])))
    if kind == "psd":
        n = 1 << (c["samples"] - 1).bit_length()
        m = masses(rng, 1)
        return dict(kind=kind, c=c, strain=noise_strain(gen, rng, n, c["fs"], c["dets"], c["samples"], 30.0, *m, 1, 4))
    if kind == "bank":
        n, fs = 1 << c["lg"], c["fs"]
        p = mf.Plan(fs, n, 1, 30.0, fs / 2, 5.5, int(fs), dtype=DTYPE[c["bank"]])
        p.set_psd(psd_bins(n, fs))
        p.bank_reserve(c["tmpl"], DTYPE[c["bank"]])
        return dict(kind=kind, c=c, plan=p, m=masses(rng, c["tmpl"]))
    if kind == "proposal":
        B, n_out = c["batch"], c["slots"]
        net = mf.MLP(5, c["width"], c["depth"], n_out, B)
        theta, d = [], 5
        for layer in range(c["depth"] + 1):
            o = c["width"] if layer < c["depth"] else n_out
            theta += [rng.standard_normal(d * o) * math.sqrt(2.0 / d), 0.01 * rng.standard_normal(o)]
            d = o
        theta = np.concatenate(theta).astype(np.float32)
        net.set_params(theta)
        nv = np.maximum(1, (n_out * rng.uniform(0.02, 1.0, B) ** 2)).astype(np.int32)
        s = dict(kind=kind, c=c, net=net, theta=theta,
                 x=torch.from_numpy(rng.standard_normal((B, 5)).astype(np.float32)).to(DEV),
                 n_valid=torch.from_numpy(nv).to(DEV),
                 label=torch.from_numpy((rng.random(B) ** 2 * nv).astype(np.int32)).to(DEV))
        s["loss"] = torch.zeros(1, device=DEV)
        s["grad"] = torch.zeros(net.n_params, device=DEV)
        s["logits"] = torch.zeros((B, n_out), device=DEV)
        s["slots"] = torch.zeros((B, c["k"]), dtype=torch.int32, device=DEV)
        s["taken"] = torch.zeros(B, dtype=torch.int32, device=DEV)
        return s
    raise ValueError(kind)


# -- one pass -----------------------------------------------------------------------

def columns(rec, names):
    return {k: rec[k] for k in names}


def records(dtype, cap):
    """A page-locked host buffer of a fixed number of records, zeros, as a program that reads every pass keeps one."""
    return torch.zeros(cap * dtype.itemsize, dtype=torch.uint8).pin_memory().numpy().view(dtype)


def read(fn, handle, rec, names):
    """The records found, into the program's buffer (mf_get_triggers, mf_get_coincs, mf_batch_get_triggers)."""
    n = ctypes.c_int64(0)
    st = fn(handle, rec.ctypes.data, len(rec), ctypes.byref(n))
    if st not in (mf.MF_OK, mf.MF_EOVERFLOW):
        raise mf.MFError(st, "read")
    return dict(columns(rec, names), found=n.value)


def capacity(windows, thr):
    """Room for the triggers of so many windows: above what noise and the signals put over the threshold."""
    share = 0.9 if thr < 4 else 0.5 if thr < 4.5 else 0.2 if thr < 5 else 0.08
    return int(min(1 << 20, max(256, share * windows)))


TRIG = ("det", "tmpl", "sample", "snr", "phase")
COINC = ("tmpl", "shift", "sample0", "sample1", "snr0", "snr1", "rho_c")


def run(s):
    c, kind = s["c"], s["kind"]
    if kind == "segment":
        s["plan"].strain_to_fd(s["strain"], s["d"])
        s["plan"].filter(s["d"])
        return dict(spectrum=s["d"], trig=read(mf.load().mf_get_triggers, s["plan"].h, s["rec"], TRIG))
    if kind == "filter":
        s["plan"].filter(s["d"], subset=s["sel"])
        return read(mf.load().mf_get_triggers, s["plan"].h, s["rec"], TRIG)
    if kind == "stage1":
        p = s["plan"]
        p.filter(s["d"])
        p.coincide(s["followed"], c["shift"], c["shifts"], int(0.015 * c["fs"]), c["rho_c"])
        return dict(coincs=read(mf.load().mf_get_coincs, p.h, s["rec"], COINC), followed=s["followed"])
    if kind == "veto":
        chi2, newsnr, sg, hat = s["out"]
        s["plan"].chisq(c["bands"], chi2, newsnr)
        s["plan"].sgchisq(s["f_final"], s["mtotal"], newsnr, sg, hat)
        return [v[:s["cap"]] for v in s["out"]]
    if kind == "hierarchy":
        h = s["h"]
        with torch.cuda.stream(h.stream):
            h.strain.copy_(s["strain"], non_blocking=True)
        union = h.run()
        co = read(mf.load().mf_get_coincs, h.p1.h, s["co"], COINC)
        return dict(trig=read(mf.load().mf_get_triggers, h.p2.h, s["rec"], TRIG), coincs=co, union=union)
    if kind == "batch":
        s["b"].run(s["strain"])
        return read(mf.load().mf_batch_get_triggers, s["b"].h, s["rec"], ("cls",) + TRIG)
    if kind == "psd":
        return mf.psd_welch(s["strain"], c["fs"], 1 << c["lg"], c["stride"], c["average"])
    if kind == "bank":
        s["plan"].bank_generate_taylorf2(0, s["m"][0], s["m"][1], 30.0)
        return s["plan"].sigmasq()
    if c["train"]:
        s["net"].loss_grad(s["x"], s["n_valid"], s["label"], loss=s["loss"], grad=s["grad"])
        s["net"].adamw_step(2e-3, weight_decay=1e-4)
        return dict(loss=s["loss"], grad=s["grad"])
    s["net"].forward(s["x"], s["logits"])
    s["net"].topk(s["x"], s["n_valid"], c["k"], s["slots"], p_mass=0.9, count=s["taken"])
    return dict(logits=s["logits"], slots=s["slots"], taken=s["taken"])


# -- the work that a pass cannot do without --------------------------------------------

def fft_flops(n, series):
    return 5.0 * n * math.log2(n) * series


def work(case):
    c, kind = case, case["kind"]
    if kind in ("segment", "filter", "stage1"):
        n = 1 << c["lg"]
        sel = c.get("sel", -1)
        sel = c["tmpl"] if sel < 0 else sel
        elem = 8 if c.get("bank", "f32") == "f32" else 4
        b = sel * (n // 2) * elem + c["dets"] * (n // 2) * 8 + (n // 2) * 8
        f = fft_flops(n, sel * c["dets"]) + 8.0 * (n // 2) * sel * c["dets"]
        if kind == "segment":
            b, f = b + c["dets"] * n * 4, f + fft_flops(n, c["dets"]) / 2
        return {"bytes": float(b), "flops": f}
    if kind == "veto":  # every template once, the data of the detectors, a product and a phase per bin and trigger
        n = 1 << c["lg"]
        wins = c["dets"] * c["tmpl"] * -(-n // c["window"])
        few = 0.03 if c["thr"] < 5 else 0.004  # the share of windows that hold a trigger
        return {"bytes": float((c["tmpl"] + c["dets"]) * (n // 2) * 8), "flops": 14.0 * (n // 2) * max(1.0, few * wins)}
    if kind == "hierarchy":
        n2 = 1 << c["lg"]
        n1 = n2 // 4
        sel = min(c["fine"], c["coarse"] * c["near"]) * 0.6  # about what the follow-up selects
        return {"bytes": c["coarse"] * n1 * 4.0 + sel * n2 * 4.0 + 2 * n2 * 4.0,
                "flops": fft_flops(n1, 2 * c["coarse"]) + fft_flops(n2, 2 * sel) + fft_flops(n2, 1)}
    if kind == "batch":
        n, fs = 1 << c["lg"], c["fs"]
        b, f = c["dets"] * c["secs"] * fs * 4.0, 0.0
        for L, t in zip(CLASS_LEN, [int(v) for v in c["per"].split(",")]):
            if t and L * fs < n:
                segs = math.ceil((c["secs"] - L) * fs / (n - L * fs))
                b += t * (n // 2) * 8.0
                f += fft_flops(n, (t + 0.5) * segs * c["dets"])
        return {"bytes": b, "flops": f}
    if kind == "psd":
        n = 1 << c["lg"]
        segs = (c["samples"] - n) // c["stride"] + 1
        return {"bytes": c["dets"] * (c["samples"] * 4.0 + (n // 2 + 1) * 8.0), "flops": fft_flops(n, segs * c["dets"]) / 2}
    if kind == "bank":
        n = 1 << c["lg"]
        return {"bytes": c["tmpl"] * (n // 2) * (8.0 if c["bank"] == "f32" else 4.0), "flops": 30.0 * c["tmpl"] * (n // 2)}
    w, o, B = c["width"], c["slots"], c["batch"]
    params = 5 * w + w + (c["depth"] - 1) * (w * w + w) + w * o + o
    return {"bytes": params * (4.0 * 8 if c["train"] else 2.0) + B * (0 if c["train"] else o * 4.0 + c["k"] * 4.0),
            "flops": 2.0 * B * params * (3 if c["train"] else 1)}


# -- the same in 64 bits ------------------------------------------------------------------

def exact_triggers(c, d, m1, m2, sel):
    """Window maxima over the threshold of rho = |z| / sigma, ordered by (det, selection, sample)."""
    n, fs = 1 << c["lg"], c["fs"]
    w, win = weights(n, fs, low_cut(fs)), c["window"]
    nb, n_win = n // 2 + 1, -(-n // win)
    ids = np.arange(c["tmpl"]) if sel is None else sel
    out = {k: [] for k in TRIG}
    for a in range(0, len(ids), 16):
        part = ids[a:a + 16]
        h = waveforms(n, fs, m1[part], m2[part], low_cut(fs)).to(torch.complex128)
        sigma = torch.sqrt((w * (h.real ** 2 + h.imag ** 2)).sum(dim=1))
        for j in range(c["dets"]):
            x = torch.zeros((len(part), n), dtype=torch.complex128, device=DEV)
            x[:, :nb] = w * d[j].to(torch.complex128) * h.conj()
            z = torch.fft.ifft(x, dim=-1, norm="forward") / sigma[:, None]
            r = torch.zeros((len(part), n_win * win), dtype=torch.float64, device=DEV)
            r[:, :n] = z.real ** 2 + z.imag ** 2
            top, at = r.view(len(part), n_win, win).max(dim=2)
            i, v = torch.nonzero(top >= c["thr"] ** 2, as_tuple=True)
            pos = v * win + at[i, v]
            zz = z[i, pos]
            ph = torch.remainder(torch.round((torch.angle(zz) / (2 * math.pi) + 0.5) * 2048), 2048)
            out["det"].append(torch.full_like(i, j))
            out["tmpl"].append(torch.from_numpy(part.astype(np.int64)).to(DEV)[i])
            out["sample"].append(pos)
            out["snr"].append(zz.abs())
            out["phase"].append((ph / 2048 - 0.5) * 2 * math.pi)  # in steps of 2 pi / 2048, as it is kept
    out = {k: torch.cat(v) for k, v in out.items()}
    place = {int(t): i for i, t in enumerate(ids)}
    at = torch.tensor([place[int(t)] for t in out["tmpl"].tolist()], dtype=torch.int64, device=DEV)
    order = torch.argsort((out["det"] * len(ids) + at) * n + out["sample"])
    return {k: v[order] for k, v in out.items()}


def filled(t, cap):
    """As the record buffer holds them: zeros after the last one; the whole numbers have no value in 64 bits of their own."""
    out = {k: None for k in TRIG + ("found",)}
    for k in ("snr", "phase"):
        out[k] = torch.zeros(cap, dtype=torch.float64, device=DEV)
        out[k][:len(t[k])] = t[k][:cap]
    return out


def exact_vetoes(c, d, m1, m2, t):
    n, fs, p = 1 << c["lg"], c["fs"], c["bands"]
    w, nb, df = weights(n, fs, low_cut(fs)), n // 2 + 1, c["fs"] / n
    k = torch.arange(nb, device=DEV)
    f = k.to(torch.float64) * df
    chi2, new, sg, hat = (torch.zeros(len(t["det"]), dtype=torch.float64, device=DEV) for _ in range(4))
    det, tm, at, rho = (t[x].tolist() for x in ("det", "tmpl", "sample", "snr"))
    last, fin = -1, f_isco(m1, m2)
    for i in sorted(range(len(det)), key=lambda v: tm[v]):
        if tm[i] != last:
            last = tm[i]
            h = waveforms(n, fs, m1[last:last + 1], m2[last:last + 1], low_cut(fs))[0].to(torch.complex128)
            power = w * (h.real ** 2 + h.imag ** 2)
            sigma2 = power.sum()
            band = torch.clamp(torch.floor(p * (torch.cumsum(power, 0) - power) / sigma2), 0, p - 1).to(torch.int64)
        ang = torch.remainder(k * at[i], n).to(torch.float64) * (2 * math.pi / n)
        q = w * d[det[i]].to(torch.complex128) * torch.polar(torch.ones_like(ang), ang)
        x = q * h.conj()
        z = torch.zeros((p, 2), dtype=torch.float64, device=DEV).index_add_(0, band, torch.view_as_real(x))
        c2 = p * ((z - z.sum(0) / p) ** 2).sum() / sigma2
        cr = c2 / (2 * p - 2)
        chi2[i], new[i] = c2, rho[i] / max(1.0, float((1 + cr ** 3) / 2)) ** (1.0 / 6)
        hat[i] = new[i]
        if m1[last] + m2[last] > 30.0:
            total, used = 0.0, 0
            for off in (15.0, 30.0, 45.0, 60.0, 75.0, 90.0, 105.0, 120.0):
                f0 = float(fin[last]) + off
                if f0 < fs / 2:
                    g = torch.exp(-(math.pi * 20.0 / (math.sqrt(2.0) * math.pi * f0) * (f - f0)) ** 2)
                    zz, s2 = (q * g).sum(), float((w * g * g).sum())
                    if s2 > 0:
                        total, used = total + float(zz.abs() ** 2) / s2, used + 1
            if used:
                sg[i] = total / (2 * used)
                if sg[i] >= 6:
                    hat[i] = new[i] / torch.sqrt(sg[i])
    return [chi2, new, sg, hat]


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("segment", "filter", "veto"):
        # Lists hold the same triggers in 64 bits where the filter keeps FP32 throughout and few are near the
        # threshold; one that is in only one of two lists would move all that follow it.
        if "f16" in (c.get("bank"), c.get("inter")) or c.get("bank") == "bf16" or c["thr"] < 4.5:
            return None
        m1, m2, d, sel = search_inputs(c, seed)
        wins = (c["tmpl"] if sel is None else c["sel"]) * c["dets"] * -(-(1 << c["lg"]) // c["window"])
        cap = capacity(wins, c["thr"])
        if kind == "segment":  # from the strain that the call is given
            n, fs = 1 << c["lg"], c["fs"]
            strain = (torch.fft.irfft(d.to(torch.complex128), n=n, dim=-1) * fs).to(torch.float32)
            d = torch.fft.rfft(strain.to(torch.float64), dim=-1) / fs
            return dict(spectrum=d, trig=filled(exact_triggers(c, d, m1, m2, None), cap))
        t = exact_triggers(c, d, m1, m2, sel)
        if kind == "filter":
            return filled(t, cap)
        if len(t["det"]) > min(cap, 12000):
            return None
        return [torch.nn.functional.pad(v, (0, cap - len(v))) for v in exact_vetoes(c, d, m1, m2, t)]
    if kind == "psd":
        s = prepare(c, seed)["strain"].to(torch.float64)
        n, fs = 1 << c["lg"], c["fs"]
        x = s.unfold(1, n, c["stride"])
        win = 0.5 - 0.5 * torch.cos(2 * math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n)
        pw = torch.cat([torch.fft.rfft(win * x[:, a:a + 64], dim=-1).abs() ** 2 for a in range(0, x.shape[1], 64)], dim=1)
        pw = 2.0 * pw / (fs * (win * win).sum())
        pw[..., 0] /= 2
        pw[..., -1] /= 2
        if c["average"] == "mean":
            return pw.mean(dim=1)
        m = x.shape[1]
        v = torch.sort(pw, dim=1).values
        med = v[:, m // 2] if m % 2 else 0.5 * (v[:, m // 2 - 1] + v[:, m // 2])
        return med / (1.0 + sum(1.0 / (2 * i + 1) - 1.0 / (2 * i) for i in range(1, (m - 1) // 2 + 1)))
    if kind == "bank":
        n, fs = 1 << c["lg"], c["fs"]
        m1, m2 = masses(rngs(seed + 7)[0], c["tmpl"])
        f = torch.arange(n // 2 + 1, dtype=torch.float64, device=DEV) * (fs / n)
        f[0] = 1.0
        below = torch.cumsum(weights(n, fs, 30.0) * f.pow(-7.0 / 3.0), 0)
        last = torch.from_numpy(np.floor(np.minimum(f_isco(m1, m2), fs / 2) / (fs / n)).astype(np.int64)).to(DEV)
        return below[last]
    if kind == "proposal":
        s = prepare(c, seed)
        th = torch.from_numpy(s["theta"]).to(DEV, torch.float64).requires_grad_(True)
        h, o, d = s["x"].to(torch.float64), 0, 5
        for layer in range(c["depth"] + 1):
            e = c["width"] if layer < c["depth"] else c["slots"]
            h = h @ th[o:o + d * e].view(d, e) + th[o + d * e:o + d * e + e]
            o, d = o + d * e + e, e
            if layer < c["depth"]:
                h = torch.nn.functional.gelu(h)
        if not c["train"]:
            return dict(logits=h.detach(), slots=None, taken=None)
        dead = torch.arange(c["slots"], device=DEV)[None, :] >= s["n_valid"][:, None]
        logp = torch.log_softmax(h.masked_fill(dead, -math.inf), dim=1)
        loss = -logp.gather(1, s["label"][:, None].to(torch.int64)).mean()
        loss.backward()
        return dict(loss=loss.detach().reshape(1), grad=th.grad)
    return None  # whole calls and lists of coincidences: selections of what the other kinds return
