"""GPU check of the chi^2 bands bin by bin: data in the last bin of each band and in the first of the next one alone, so
that a bin in the wrong band changes the statistic by as much as the bin holds."""

import numpy as np
import pytest

import synth
from oracle import mf_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("lg,bands", [(12, 5), (14, 16), (17, 64)])
def test_bins_at_band_edges(lib, lg, bands):
    from paper_2309_00019_gb300 import mf
    n, fs, f_low = 1 << lg, 1024.0, 25.0
    rng = np.random.default_rng(lg)
    psd = synth.psd_bins(n, fs)
    w = O.weights(n, fs, f_low, fs / 2, psd)
    # the white template's power varies from bin to bin, so that no band edge is a tie of the running sum
    h = (rng.uniform(0.5, 1.5, len(w)) * np.exp(2j * np.pi * rng.random(len(w))) / np.sqrt(np.where(w > 0, w, 1.0)))
    h = np.where(w > 0, h, 0).astype(np.complex64)
    band = O.chisq_bins(h.astype(np.complex128), w, bands)
    first = np.array([np.flatnonzero(band == l)[0] for l in range(1, bands)])
    last = np.array([np.flatnonzero(band == l)[-1] for l in range(bands - 1)])
    s = np.zeros((1, len(w)), np.complex64)
    for k in np.concatenate([first, last]):
        s[0, k] = 8.0 * np.exp(2j * np.pi * rng.random()) * abs(h[k]) * np.sqrt(O.sigmasq(h, w)) / (w[k] * abs(h[k]) ** 2)
    p = mf.Plan(fs, n, 1, f_low, fs / 2, 3.0, n // 16, max_triggers=64)
    p.set_psd(psd)
    p.load_bank(torch.from_numpy(h[None]).to(DEV))
    p.filter(torch.from_numpy(s).to(DEV))
    trig, count, _ = p.triggers()
    assert count == len(trig) == 16
    chi2, new = torch.zeros(64, device=DEV), torch.zeros(64, device=DEV)
    p.chisq(bands, chi2, new)
    torch.cuda.synchronize()
    s64, h64 = s[0].astype(np.complex128), h.astype(np.complex128)
    for i, t in enumerate(trig):
        ref = O.chisq(s64, h64, w, n, int(t["sample"]), bands)
        # each bin adds 8 to |z| / sigma: p sum |z_l|^2 / sigma^2 <= p (bands - 1) 16^2.  A term's FP32 operations (weighted
        # data, product, two phases and their products, sum) are right to 12 roundings of 2^-24, its square to twice that
        assert abs(float(chi2[i]) - ref) <= 24 * 2.0 ** -24 * bands * (bands - 1) * 256, (i, chi2[i], ref)
