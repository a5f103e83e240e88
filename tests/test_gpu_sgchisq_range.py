"""GPU check of the sine-Gaussian veto's tiles that hold no bin: frequencies so far below zero that their first or last
bin passes 32 bits (with the usual quality and with one whose tiles are wider than their frequency), infinite and not a
number.  They are left out: a trigger with such tiles alone keeps its SNR."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("q", [20.0, 5.0])
@pytest.mark.parametrize("f", [-200.0, -1.5e7, -6.0e7, -1.2e8, -1.0e30, -np.inf, np.nan])
def test_tiles_without_bins(lib, f, q):
    from paper_2309_00019_gb300 import mf
    n, fs, cap = 1 << 16, 2048.0, 1 << 10
    rng = np.random.default_rng(3)
    p = mf.Plan(fs, n, 1, 30.0, fs / 2, 3.0, 2048, max_triggers=cap)
    p.set_psd(synth.psd_bins(n, fs))
    p.load_bank(synth.taylorf2_torch(n, fs, np.array([25.0, 40.0]), np.array([20.0, 30.0]), 30.0, DEV))
    p.filter(torch.from_numpy(synth.coloured_noise_fd(rng, n, fs).astype(np.complex64)[None]).to(DEV))
    _, count, _ = p.triggers()
    assert 0 < count <= cap
    snr = torch.from_numpy(rng.uniform(4, 9, cap).astype(np.float32)).to(DEV)
    c2, hat = torch.full((cap,), -1.0, device=DEV), torch.full((cap,), -1.0, device=DEV)
    p.sgchisq(torch.full((2,), f, device=DEV), torch.full((2,), 60.0, device=DEV), snr, c2, hat, q=q)
    torch.cuda.synchronize()
    assert not c2[:count].any() and torch.equal(hat[:count], snr[:count])
