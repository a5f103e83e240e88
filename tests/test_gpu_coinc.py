"""GPU checks of the coincidences over shapes against a walk over all pairs and shifts on the filter's own triggers:
few and many windows, shifts that wrap the ring, shifts that meet the coincidence window, one shift, a step that is
a multiple of the ring, records in order, and more records than a template's collection holds."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def mf(lib):
    from paper_2309_00019_gb300 import mf as m
    return m


@pytest.mark.parametrize("lg,window,valid,shift,shifts,cw,rho_c", [
    (14, 512, (0, 1 << 14), 640, 20, 7, 5.0),            # shifts within the ring
    (14, 200, (1000, 15001), 3001, 40, 30, 5.5),         # ragged windows, shifts that wrap several times
    (13, 64, (0, 1 << 13), 5, 9, 16, 5.0),               # steps below the coincidence window: several shifts per pair
    (13, 128, (0, 1 << 13), 1 << 13, 3, 5, 4.5),         # every shift is a whole turn
    (12, 1, (0, 1 << 12), 100, 12, 4, 4.6),              # a window per sample: the walk over windows
    (13, 32, (16, 8000), 777, 0, 40, 4.2),               # zero lag only, low threshold
    (14, 16, (0, 1 << 14), 50, 60, 25, 4.4),             # many records per template
])
def test_coincidences_over_shapes(mf, lg, window, valid, shift, shifts, cw, rho_c):
    n, fs, f_low, tmpl = 1 << lg, 512.0, 30.0, 5
    rng = np.random.default_rng(lg + window)
    bank = np.stack([synth.taylorf2(n, fs, 2.0 + i, 1.5 + i, f_low) for i in range(tmpl)]).astype(np.complex64)
    sfd = np.stack([synth.coloured_noise_fd(rng, n, fs) for _ in range(2)]).astype(np.complex64)
    p = mf.Plan(fs, n, 2, f_low, fs / 2, 2.5, window, valid_begin=valid[0], valid_end=valid[1])
    p.set_psd(synth.psd_bins(n, fs))
    p.load_bank(torch.from_numpy(bank).to(DEV))
    sel = torch.tensor([0, 2, 3, 4], dtype=torch.int32, device=DEV)
    p.filter(torch.from_numpy(sfd).to(DEV), subset=sel)
    trig, _, _ = p.triggers()
    followed = torch.full((tmpl,), 7, dtype=torch.int32, device=DEV)
    p.coincide(followed, shift, shifts, cw, rho_c, rho_c_store=rho_c * 0.95)
    co, found, _ = p.coincs()
    want, free, follow, loose = [], set(), np.zeros(tmpl, np.int32), np.zeros(tmpl, bool)
    R = valid[1] - valid[0]
    for t in (0, 2, 3, 4):
        a, b = (trig[(trig["det"] == d) & (trig["tmpl"] == t)] for d in (0, 1))
        d = (a["sample"][:, None] - b["sample"][None, :]).astype(np.int64)
        r2 = a["snr"].astype(np.float64)[:, None] ** 2 + b["snr"].astype(np.float64)[None, :] ** 2
        # the triggers' SNRs are rounded squares' roots: rho_c^2 within 3 roundings of a threshold may fall either way
        at_thr, at_store = np.abs(r2 / rho_c ** 2 - 1) < 5e-7, np.abs(r2 / (0.95 * rho_c) ** 2 - 1) < 5e-7
        for k in range(shifts + 1):
            x = np.mod(d - k * shift, R)
            near = np.minimum(x, R - x) <= cw
            name = lambda m: [(t, k, int(a["sample"][i]), int(b["sample"][j])) for i, j in zip(*np.nonzero(m))]  # noqa: E731
            want += name(near & (r2 >= (0.95 * rho_c) ** 2) & ~at_store)
            free |= set(name(near & at_store))
            follow[t] |= int((near & (r2 >= rho_c ** 2) & ~at_thr).any())
            loose[t] |= (near & at_thr).any()
    got = list(zip(*(co[f].tolist() for f in ("tmpl", "shift", "sample0", "sample1"))))
    assert found == len(got) and len(want) > 0 and len(free) <= 2
    assert got == sorted(got) and [g for g in got if g not in free] == sorted(want)
    flags = followed.cpu().numpy()
    assert all(flags[t] == follow[t] or loose[t] for t in range(tmpl))
    few, count, _ = p.coincs(cap=3)
    assert count == found and np.array_equal(few, co[:3])
