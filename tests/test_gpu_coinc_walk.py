"""GPU checks of the coincidences where most triggers are loud, which walk over the shifts of each detector-0 trigger: up to
2,048 windows, shift counts around the piece that a thread walks, several turns of a ragged ring, no and a wide
coincidence window, and a selection, against all pairs and shifts of the filter's own triggers."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("lg,window,valid,shift,shifts,cw,rho_c,store", [
    (12, 2, (0, 1 << 12), 1, 0, 8, 1.0, 4.3),          # 2,048 windows, zero lag
    (13, 4, (0, 1 << 13), 700, 63, 2, 1.0, 5.2),       # one piece of shifts
    (13, 4, (0, 1 << 13), 701, 64, 0, 1.0, 4.6),       # a piece and one shift, exact times only
    (12, 3, (101, 3998), 1500, 130, 5, 1.0, 5.4),      # ragged windows and ring, many turns
    (12, 5, (7, 4096), 4089 * 2, 3, 3, 1.0, 4.4),      # whole turns
    (14, 64, (0, 1 << 14), 90, 20, 3000, 4.4, 5.9),    # a coincidence window of many windows
    (14, 64, (500, 16000), 511, 2, 20, 5.5, 4.0),      # followed above what is stored
    (14, 64, (500, 16000), 511, 2, 20, 4.0, 5.5),      # and below
])
def test_most_triggers_loud(lib, lg, window, valid, shift, shifts, cw, rho_c, store):
    from paper_2309_00019_gb300 import mf
    n, fs, f_low, tmpl = 1 << lg, 512.0, 30.0, 4
    rng = np.random.default_rng(lg + window + cw)
    bank = np.stack([synth.taylorf2(n, fs, 2.0 + i, 1.5 + i, f_low) for i in range(tmpl)]).astype(np.complex64)
    sfd = np.stack([synth.coloured_noise_fd(rng, n, fs) for _ in range(2)]).astype(np.complex64)
    p = mf.Plan(fs, n, 2, f_low, fs / 2, 1.5, window, valid_begin=valid[0], valid_end=valid[1])
    p.set_psd(synth.psd_bins(n, fs))
    p.load_bank(torch.from_numpy(bank).to(DEV))
    ids = [3, 0, 2]
    p.filter(torch.from_numpy(sfd).to(DEV), subset=torch.tensor(ids, dtype=torch.int32, device=DEV))
    trig, _, _ = p.triggers()
    followed = torch.full((tmpl,), 7, dtype=torch.int32, device=DEV)
    p.coincide(followed, shift, shifts, cw, rho_c, rho_c_store=store)
    co, found, _ = p.coincs()
    got = list(zip(*(co[f].tolist() for f in ("tmpl", "shift", "sample0", "sample1"))))
    want, free = [], set()
    follow, loose = np.zeros(tmpl, np.int32), np.zeros(tmpl, bool)
    R = valid[1] - valid[0]
    for t in ids:
        a, b = (trig[(trig["det"] == d) & (trig["tmpl"] == t)] for d in (0, 1))
        d = (a["sample"][:, None] - b["sample"][None, :]).astype(np.int32)
        r2 = a["snr"].astype(np.float64)[:, None] ** 2 + b["snr"].astype(np.float64)[None, :] ** 2
        # the triggers' SNRs are rounded squares' roots: rho_c^2 within 3 roundings of a threshold may fall either way
        at_thr, at_store = np.abs(r2 / rho_c ** 2 - 1) < 5e-7, np.abs(r2 / store ** 2 - 1) < 5e-7
        for k in range(shifts + 1):
            x = np.mod(d - np.int32(k * shift % R), np.int32(R))
            near = np.minimum(x, R - x) <= cw
            name = lambda m: [(t, k, int(a["sample"][i]), int(b["sample"][j])) for i, j in zip(*np.nonzero(m))]  # noqa: E731
            want += name(near & (r2 >= store ** 2) & ~at_store)
            free |= set(name(near & at_store))
            follow[t] |= int((near & (r2 >= rho_c ** 2) & ~at_thr).any())
            loose[t] |= (near & at_thr).any()
    assert found == len(got) and len(want) > 0 and len(free) <= 2
    assert got == sorted(got) and [g for g in got if g not in free] == sorted(want)
    flags = followed.cpu().numpy()
    assert all(flags[t] == follow[t] or loose[t] for t in range(tmpl))
