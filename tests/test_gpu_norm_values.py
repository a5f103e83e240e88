"""The norm's squares are put together from the bits of the stored values: rows of every kind of value (subnormal,
smallest normal, largest, mixed with zeros in one part) against FP64 sums."""

import numpy as np
import pytest

import synth
from oracle import mf_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def test_norms_of_all_kinds_of_values(lib):
    from paper_2309_00019_gb300 import mf
    n, fs = 1 << 12, 1024.0
    nb = n // 2 + 1
    rng = np.random.default_rng(5)

    def values(lo, hi, subnormal=False):  # random bits with exponents in [lo, hi]
        e = np.zeros(nb, np.uint32) if subnormal else rng.integers(lo, hi + 1, nb).astype(np.uint32)
        u = (rng.integers(0, 2, nb).astype(np.uint32) << 31) | (e << 23) | rng.integers(0, 1 << 23, nb).astype(np.uint32)
        return u.view(np.float32)

    rows = []
    for re, im in [(values(1, 1), values(1, 1)), (values(254, 254), values(250, 254)), (values(1, 254), values(1, 254)),
                   (values(0, 0, True), values(0, 0, True)), (values(0, 0, True), values(1, 4)),
                   (np.zeros(nb, np.float32), values(120, 130)), (values(120, 130), np.zeros(nb, np.float32)),
                   (np.full(nb, 1.0, np.float32), np.full(nb, np.float32(np.sqrt(2.0)), np.float32))]:
        rows.append((re + 1j * im).astype(np.complex64))
    h = np.stack(rows)
    h[2, rng.integers(0, nb, nb // 3)] = 0
    psd = synth.psd_bins(n, fs)
    w = O.weights(n, fs, 20.0, fs / 2, psd)
    p = mf.Plan(fs, n, 1, 20.0, fs / 2, 5.0, n, max_triggers=16)
    p.set_psd(psd)
    p.bank_reserve(len(h))
    p.bank_set_rows(0, torch.from_numpy(h).to(DEV))
    # sums of n/2 positive FP64 terms in any order: n/2 x 2^-53 at most
    assert np.allclose(p.sigmasq(), O.sigmasq(h.astype(np.complex128), w), rtol=n * 2.0 ** -54 + 2.0 ** -51, atol=0)
