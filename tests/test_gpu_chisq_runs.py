"""The chi^2 veto of long trigger lists, whose triggers share their loads in runs of up to eight (four where a row has
1,024 bins), against the same triggers in lists short enough for one trigger at a time."""

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


def veto(mf, n, bank, sfd, psd, window, fmt, cap):
    fs, f_low = 1024.0, 25.0
    p = mf.Plan(fs, n, len(sfd), f_low, fs / 2, 1.0, window, max_triggers=cap, dtype=getattr(mf, fmt))
    p.set_psd(psd)
    p.load_bank(torch.from_numpy(bank).to(DEV))
    p.filter(torch.from_numpy(sfd).to(DEV))
    trig, count, _ = p.triggers()
    assert count == len(trig)
    chi2, new = torch.zeros(cap, device=DEV), torch.zeros(cap, device=DEV)
    p.chisq(8, chi2, new)
    torch.cuda.synchronize()
    return trig, chi2.cpu().numpy()[:count], new.cpu().numpy()[:count]


# (nearly every window crosses so low a threshold)
@pytest.mark.parametrize("lg,tmpl,windows,fmt", [(12, 260, 10, "MF_F32"), (14, 250, 11, "MF_F16"), (16, 170, 17, "MF_F32"),
                                                 (20, 20, 128, "MF_F32")])
def test_runs_of_long_lists(mf, lg, tmpl, windows, fmt):
    n, fs = 1 << lg, 1024.0
    rng = np.random.default_rng(lg)
    bank = np.stack([synth.taylorf2(n, fs, 3.0 + 0.01 * i, 1.5, 25.0) for i in range(tmpl)]).astype(np.complex64)
    sfd = np.stack([synth.coloured_noise_fd(rng, n, fs) for _ in range(2)]).astype(np.complex64)
    psd = synth.psd_bins(n, fs)
    window = -(-n // windows)
    trig, chi2, new = veto(mf, n, bank, sfd, psd, window, fmt, 1 << 14)
    assert len(trig) > 8 * 4 * 152  # eight triggers and more for each block of the largest grid
    for t in (0, tmpl // 2, tmpl - 1):
        one, c1, n1 = veto(mf, n, bank[t:t + 1], sfd, psd, window, fmt, 1 << 14)
        mine = trig["tmpl"] == t
        assert np.array_equal(one["sample"], trig["sample"][mine]) and len(one) < 4 * 152
        # the same FP32 products in the same order for each trigger: differences are roundings of the turned sums,
        # 2^-23 of the largest of 8 band sums, whose squares make chi^2 <= 100
        assert np.abs(chi2[mine] - c1).max() <= 1e-4 * max(1.0, float(c1.max()))
        assert np.abs(new[mine] - n1).max() <= 1e-4 * float(n1.max())
