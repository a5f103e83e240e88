"""GPU parity of the chi^2 veto over shapes: pieces of rows (small N) and several rows per thread (N = 2^20), band
counts whose edges share pieces or leave bands empty, and runs of 1, 2, 3, 4 and more triggers per template."""

import numpy as np
import pytest

import synth
from oracle import mf_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def mf(lib):
    from paper_2309_00019_gb300 import mf as m
    return m


@pytest.mark.parametrize("lg,bands,tmpl,window", [(12, 2, 5, 256), (13, 64, 3, 128), (14, 13, 4, 512), (16, 64, 2, 2048),
                                                  (19, 7, 2, 1 << 14), (20, 16, 2, 1 << 15)])
def test_chisq_over_shapes(mf, lg, bands, tmpl, window):
    n, fs, f_low = 1 << lg, 1024.0, 25.0
    rng = np.random.default_rng(lg + bands)
    bank = np.stack([synth.taylorf2(n, fs, 3.0 + i, 1.5 + i, f_low) for i in range(tmpl)]).astype(np.complex64)
    # narrow lines: most of a template's power in few bins, so that bands end next to each other and some are empty
    bank[0, n // 9: n // 9 + 3] *= 40.0
    sfd = np.stack([synth.coloured_noise_fd(rng, n, fs) for _ in range(2)])
    psd = synth.psd_bins(n, fs)
    p = mf.Plan(fs, n, 2, f_low, fs / 2, 3.0, window, max_triggers=4096)
    p.set_psd(psd)
    p.load_bank(torch.from_numpy(bank).to(DEV))
    p.filter(torch.from_numpy(sfd.astype(np.complex64)).to(DEV))
    trig, count, _ = p.triggers()
    assert count == len(trig) > tmpl
    chi2, new = torch.zeros(4096, device=DEV), torch.zeros(4096, device=DEV)
    p.chisq(bands, chi2, new)
    torch.cuda.synchronize()
    chi2, new = chi2.cpu().numpy(), new.cpu().numpy()
    assert not chi2[count:].any() and not new[count:].any()
    w = O.weights(n, fs, f_low, fs / 2, psd)
    for i in np.unique(np.linspace(0, count - 1, 24).astype(int)):
        t = trig[i]
        ref = O.chisq(sfd[t["det"]].astype(np.complex64).astype(np.complex128), bank[t["tmpl"]].astype(np.complex128), w,
                      n, int(t["sample"]), bands)
        # FP32 products and row sums: the same bound as on the other shapes of this veto
        assert abs(float(chi2[i]) - ref) <= 2e-3 * max(ref, 1.0), (i, t, chi2[i], ref)
        exp = float(O.newsnr(float(t["snr"]), O.reduced_chisq(ref, bands)))
        assert new[i] == pytest.approx(exp, rel=2e-3, abs=1e-5)
