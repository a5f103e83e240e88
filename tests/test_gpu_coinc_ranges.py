"""GPU check that the coincidences of a filter whose rows had analysed ranges of their own do not depend on what the plan's
ranges are when they are asked for: triggers outside the plan's ring, the ranges kept, taken away, or set after a filter
without them."""

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def test_ranges_are_those_of_the_filter(lib):
    from paper_2309_00019_gb300 import mf
    n, fs, f_low, tmpl = 1 << 14, 512.0, 30.0, 4
    rng = np.random.default_rng(9)
    bank = np.stack([synth.taylorf2(n, fs, 2.0 + i, 1.5 + i, f_low) for i in range(tmpl)]).astype(np.complex64)
    data = torch.from_numpy(np.stack([synth.coloured_noise_fd(rng, n, fs) for _ in range(2)]).astype(np.complex64)).to(DEV)
    wide = np.array([[0, n], [0, n]])
    # a ring that is a small part of the rows' ranges: most times are outside it, some by several turns
    p = mf.Plan(fs, n, 2, f_low, fs / 2, 2.5, 200, valid_begin=9000, valid_end=11000)
    p.set_psd(synth.psd_bins(n, fs))
    p.load_bank(torch.from_numpy(bank).to(DEV))

    def coincs():
        followed = torch.full((tmpl,), 7, dtype=torch.int32, device=DEV)
        p.coincide(followed, 311, 30, 20, 4.5, rho_c_store=4.0)
        return p.coincs()[0], followed.cpu().numpy()

    p.set_row_valid(wide)
    p.filter(data)
    t = p.triggers()[0]
    assert (t["sample"] < 9000).any() and (t["sample"] >= 11000).any()
    kept, f0 = coincs()
    p.set_row_valid(None)
    gone, f1 = coincs()
    assert len(kept) > 0 and np.array_equal(kept, gone) and np.array_equal(f0, f1)
    p.filter(data)
    plain, f0 = coincs()
    p.set_row_valid(wide)
    late, f1 = coincs()
    assert len(plain) > 0 and np.array_equal(plain, late) and np.array_equal(f0, f1)
