"""GPU checks of coincidence counts that pass the per-template collection and 32 bits: a shift of a whole turn, so that
every pair in reach coincides at all of millions of shifts, and runs of neighbouring shifts, against a count over pairs."""

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


@pytest.mark.parametrize("window,shift,shifts,cw,wide", [
    (64, 1 << 12, (1 << 22) - 3, 400, True),  # 64 windows each: some 800 pairs in reach, 4,194,302 shifts of each
    (64, 1 << 12, 600, 400, False),           # runs longer than the collection
    (16, 1, 300, 3, False),                   # runs of seven shifts, many more than the collection holds
    (16, 1, 40, 4, False),                    # runs of nine
])
def test_counts_past_the_collection(mf, window, shift, shifts, cw, wide):
    n, fs, rho, cap = 1 << 12, 1024.0, 0.5, 1 << 20
    rng = np.random.default_rng(window)
    p = mf.Plan(fs, n, 2, 25.0, fs / 2, 0.6, window)
    p.set_psd(synth.psd_bins(n, fs))
    p.load_bank(torch.from_numpy(synth.taylorf2(n, fs, 3.0, 1.5, 25.0).astype(np.complex64)[None]).to(DEV))
    p.filter(torch.from_numpy(np.stack([synth.coloured_noise_fd(rng, n, fs) for _ in range(2)]).astype(np.complex64)).to(DEV))
    trig, _, _ = p.triggers()
    a, b = (trig["sample"][trig["det"] == d].astype(np.int64) for d in (0, 1))
    # the ring distance d - k shift, for every pair; the thresholds are below every pair's combined SNR
    d = np.mod(a[:, None] - b[None, :], n)
    k = np.arange(min(shifts + 1, n))  # the distances repeat after a turn
    x = np.mod(d[..., None] - (k * shift)[None, None, :], n) if not wide else d[..., None]
    want = int((np.minimum(x, n - x) <= cw).sum()) * (shifts + 1 if wide else 1)
    assert (want > 1 << 31) == wide and want > 512
    followed = torch.zeros(1, dtype=torch.int32, device=DEV)
    p.coincide(followed, shift, shifts, cw, rho, max_coincs=cap)
    co, found, st = p.coincs(cap=cap)
    assert found == want and len(co) == min(want, cap) and followed.item() == 1
    y = np.mod(co["sample0"] - co["sample1"] - co["shift"].astype(np.int64) * shift, n)
    assert (np.minimum(y, n - y) <= cw).all() and (co["shift"] >= 0).all() and (co["shift"] <= shifts).all()
    assert len(np.unique(co[["shift", "sample0", "sample1"]])) == len(co)
