"""GPU checks of the coincidences over the shapes of the launch: threads by windows, a template's detector-0 triggers shared
among CTAs, or CTAs that take several windows per thread; pairs and walks; and what a call may take."""

import time

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def plan(lib, lg, window, thr, tmpl):
    from paper_2309_00019_gb300 import mf
    n, fs, f_low = 1 << lg, 512.0, 30.0
    rng = np.random.default_rng(lg + tmpl)
    p = mf.Plan(fs, n, 2, f_low, fs / 2, thr, window)
    p.set_psd(synth.psd_bins(n, fs))
    p.bank_reserve(tmpl)
    p.bank_generate_taylorf2(0, rng.uniform(1.2, 10, tmpl), rng.uniform(1.2, 10, tmpl), f_low)
    sfd = np.stack([synth.coloured_noise_fd(rng, n, fs) for _ in range(2)]).astype(np.complex64)
    p.filter(torch.from_numpy(sfd).to(DEV))
    return p


@pytest.mark.parametrize("lg,window,thr,tmpl", [(12, 32, 2.0, 700), (12, 31, 2.0, 3), (12, 8, 2.0, 9), (12, 4, 2.5, 330),
                                                (12, 4, 2.5, 160), (12, 4, 2.5, 2), (12, 2, 3.0, 310), (12, 2, 3.0, 155),
                                                (12, 2, 3.0, 70)])
@pytest.mark.parametrize("shift,shifts,cw,rho", [(700, 3, 9, 1.1), (1234, 30, 2, 1.6), (3, 200, 1, 1.9)])
def test_shapes_of_the_launch(lib, lg, window, thr, tmpl, shift, shifts, cw, rho):
    p = plan(lib, lg, window, thr, tmpl)
    trig, _, _ = p.triggers()
    followed = torch.zeros(tmpl, dtype=torch.int32, device=DEV)
    R, store = 1 << lg, rho * thr
    p.coincide(followed, shift, shifts, cw, store, max_coincs=1 << 22)
    co, found, _ = p.coincs()
    assert found == len(co)
    for t in sorted({0, tmpl // 2, tmpl - 1}):
        a, b = (trig[(trig["det"] == d) & (trig["tmpl"] == t)] for d in (0, 1))
        r2 = a["snr"].astype(np.float64)[:, None] ** 2 + b["snr"].astype(np.float64)[None, :] ** 2
        # the triggers' SNRs are rounded squares' roots: rho_c^2 within 3 roundings of the threshold may fall either way
        tie = np.abs(r2 / store ** 2 - 1) < 5e-7
        d = (a["sample"][:, None] - b["sample"][None, :]).astype(np.int64)
        want, free = [], set()
        for k in range(shifts + 1):
            x = np.mod(d - k * shift, R)
            near = np.minimum(x, R - x) <= cw
            for m, to in ((near & (r2 >= store ** 2) & ~tie, want.append), (near & tie, free.add)):
                for i, j in zip(*np.nonzero(m)):
                    to((k, int(a["sample"][i]), int(b["sample"][j])))
        c = co[co["tmpl"] == t]
        got = list(zip(*(c[f].tolist() for f in ("shift", "sample0", "sample1"))))
        assert [g for g in got if g not in free] == sorted(want) and len(free) <= 2
        assert bool(followed[t]) == bool(want) or free


@pytest.mark.parametrize("lg,window,thr,tmpl,shift,shifts,cw,rho_c,store",
                         [(12, 2, 1.5, 1, 613, 500, 3, 3.75, 3.75), (12, 64, 3.0, 300, 613, 500, 3, 4.35, 4.35)])
def test_lanes_stay_together(lib, lg, window, thr, tmpl, shift, shifts, cw, rho_c, store):
    p = plan(lib, lg, window, thr, tmpl)
    followed = torch.zeros(tmpl, dtype=torch.int32, device=DEV)
    took = []
    for _ in range(4):
        torch.cuda.synchronize()
        t = time.perf_counter()
        p.coincide(followed, shift, shifts, cw, rho_c, rho_c_store=store)
        torch.cuda.synchronize()
        took.append(time.perf_counter() - t)
    # 15 and 5.6 ms where the lanes of a warp that had found something went on one by one; a tenth of it where they do not
    assert min(took) < 4e-3, took
