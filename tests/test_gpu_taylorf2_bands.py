"""GPU check of generated rows whose band is a small part of the row or begins in its first bins, of heavy and light
templates in one call, with anchors at every bin and far apart, and of more rows than one block: against the float64
formula, and each row against the row made alone."""

import ctypes as C

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def gen(lib, m1, m2, n, fs, f_low):
    from paper_2309_00019_gb300 import mf
    nb = n // 2 + 1
    m1, m2 = np.ascontiguousarray(m1), np.ascontiguousarray(m2)
    out = torch.full((len(m1), nb), np.nan, dtype=torch.complex64, device=DEV)
    assert lib.mf_taylorf2(m1.ctypes.data, m2.ctypes.data, len(m1), fs, n, f_low, C.c_void_p(out.data_ptr()), nb, None) == mf.MF_OK
    torch.cuda.synchronize()
    return out.cpu().numpy()


@pytest.mark.parametrize("n,fs,f_low,rows", [
    (1 << 18, 65536.0, 20.0, 70),    # bins of 0.25 Hz: an anchor per bin, 64 rows per block
    (1 << 12, 16384.0, 10.0, 9),     # bins of 4 Hz, the band from bin 3 on
    (1 << 12, 4096.0, 1.5, 5),       # from bin 2
    (1 << 13, 1024.0, 20.0, 1100),   # anchors at every second bin
    (1 << 17, 512.0, 100.0, 6),      # far apart; the band is most of the row
    (1 << 14, 1024.0, 500.0, 5),     # the band ends below its lowest frequency for the heavy ones: empty rows
])
def test_bands(lib, n, fs, f_low, rows):
    rng = np.random.default_rng(rows)
    m1, m2 = rng.uniform(1.2, 30.0, rows), rng.uniform(1.2, 10.0, rows)
    m1[0], m2[0] = 80.0, 60.0   # f_ISCO 31 Hz
    m1[-1], m2[-1] = 1.2, 1.2   # 1.8 kHz
    got = gen(lib, m1, m2, n, fs, f_low)
    for i in {0, 1, rows // 2, min(64, rows - 1), rows - 1}:
        ref = synth.taylorf2(n, fs, m1[i], m2[i], f_low)
        assert np.array_equal(got[i] != 0, ref != 0)
        # the bound on generated templates of the other tests (interpolated phase and FP32)
        assert np.abs(got[i] - ref).max() <= 2e-3 * np.abs(ref).max()
        assert np.array_equal(got[i], gen(lib, m1[i:i + 1], m2[i:i + 1], n, fs, f_low)[0])
