"""The filter's set-up, which weights and transposes the rows of several detectors in one launch, and the compaction of
the trigger list, which one CTA does up to 4,096 window slots: against plans of one detector, whose lists hold the same
numbers."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
FS, F_LOW = 1024.0, 25.0


@pytest.fixture(scope="module")
def mf(lib):
    from paper_2309_00019_gb300 import mf as m
    return m


def run(mf, n, bank, sfd, psd, window, dtype):
    p = mf.Plan(FS, n, len(sfd), F_LOW, FS / 2, 1.5, window, max_triggers=1 << 13, dtype=dtype)
    p.set_psd(psd)
    p.load_bank(torch.from_numpy(bank).to(DEV))
    p.filter(torch.from_numpy(sfd).to(DEV))
    trig, count, _ = p.triggers()
    assert count == len(trig)
    return trig


# slots = detectors x templates x windows: 512 ... 4,096 (one CTA), 4,097 and 4,100 (all of them)
@pytest.mark.parametrize("lg,n_det,tmpl,windows,dtype", [(12, 1, 2, 256, "MF_F32"), (12, 4, 4, 256, "MF_F16"),
                                                         (12, 5, 5, 164, "MF_F32"), (13, 8, 3, 64, "MF_BF16"),
                                                         (12, 1, 17, 241, "MF_F32"), (13, 2, 16, 128, "MF_F32")])
def test_rows_of_several_detectors(mf, lg, n_det, tmpl, windows, dtype):
    n = 1 << lg
    rng = np.random.default_rng(lg + n_det)
    bank = np.stack([synth.taylorf2(n, FS, 3.0 + 0.5 * i, 1.5, F_LOW) for i in range(tmpl)]).astype(np.complex64)
    sfd = np.stack([synth.coloured_noise_fd(rng, n, FS) for _ in range(n_det)]).astype(np.complex64)
    psd = synth.psd_bins(n, FS)
    window = -(-n // windows)
    assert -(-n // window) == windows
    got = run(mf, n, bank, sfd, psd, window, getattr(mf, dtype))
    assert set(got["det"]) == set(range(n_det))
    order = np.lexsort((got["sample"], got["tmpl"], got["det"]))
    assert len(np.unique(got[["det", "tmpl", "sample"]])) == len(got)
    got = got[order]
    for d in range(n_det):
        one = run(mf, n, bank, sfd[d:d + 1], psd, window, getattr(mf, dtype))
        one = one[np.lexsort((one["sample"], one["tmpl"]))]
        mine = got[got["det"] == d]
        for f in ("tmpl", "sample", "snr", "phase"):
            assert np.array_equal(mine[f], one[f]), (d, f)
