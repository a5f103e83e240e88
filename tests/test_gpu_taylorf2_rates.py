"""Generated rows at sampling rates whose bin width FP32 holds exactly (the frequency is one FP32 product) and does not
hold (an FP64 product), against the FP64 formula."""

import ctypes as C

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("n", [1 << 12, 1 << 17])
@pytest.mark.parametrize("fs,exact", [(1024.0, True), (1000.25, True), (16777215.0 / 16384, True), (1000.1, False)])
def test_rows_over_sampling_rates(lib, n, fs, exact):
    from paper_2309_00019_gb300 import mf
    df = fs / n
    assert (float(np.float32(df)) == df) == exact
    m1, m2, nb = np.array([5.0, 30.0]), np.array([3.0, 20.0]), n // 2 + 1
    out = torch.zeros((2, nb), dtype=torch.complex64, device=DEV)
    assert lib.mf_taylorf2(m1.ctypes.data, m2.ctypes.data, 2, fs, n, 20.0, C.c_void_p(out.data_ptr()), nb, None) == mf.MF_OK
    torch.cuda.synchronize()
    got = out.cpu().numpy().astype(np.complex128)
    for i in range(2):
        ref = synth.taylorf2(n, fs, m1[i], m2[i], 20.0)
        assert np.array_equal(got[i] != 0, ref != 0)
        band = ref != 0
        # exp2(-7/6 log2 f): two units of a logarithm up to 10 (2^-19 x 7/6 x ln 2 = 1.6e-6), two of exp2 (2.4e-7) and
        # 2^-21 of sine and cosine (4.8e-7)
        assert np.abs(np.abs(got[i][band]) / np.abs(ref[band]) - 1).max() <= 4e-6
