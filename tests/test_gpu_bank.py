"""GPU checks of the bank's column-layout writer and the norms it takes on the way: every segment length (one and
several tiles per CTA), every storage type, rows with empty and partly empty bands, the PSD set before and after
the rows, and rows generated in blocks."""

import numpy as np
import pytest

import synth
from oracle import mf_oracle as O
from oracle import quant_oracle as Q

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def mf(lib):
    from paper_2309_00019_gb300 import mf as m
    return m


@pytest.mark.parametrize("kind", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("lg", [12, 13, 15, 17, 20])
def test_norms_of_stored_rows(mf, lg, kind):
    n, fs, rows = 1 << lg, 1024.0, 3 if lg < 20 else 2
    dtype = {"f32": mf.MF_F32, "f16": mf.MF_F16, "bf16": mf.MF_BF16}[kind]
    rng = np.random.default_rng(lg)
    nb = n // 2 + 1
    h = (rng.standard_normal((rows, nb)) + 1j * rng.standard_normal((rows, nb))).astype(np.complex64)
    h[0, : nb // 5] = 0  # empty below and above a band whose ends are inside a tile
    h[0, nb // 2 + 3:] = 0
    h[-1] = 0
    psd = synth.psd_bins(n, fs)
    w = O.weights(n, fs, 20.0, fs / 2, psd)

    def plan(first):
        p = mf.Plan(fs, n, 1, 20.0, fs / 2, 5.0, n, dtype=dtype, max_triggers=16)
        if first:
            p.set_psd(psd)
        p.bank_reserve(rows, dtype)
        d = torch.from_numpy(h).to(DEV)
        p.bank_set_rows(0, d) if kind == "f32" else p.bank_quantize_rows(0, d)
        if not first:
            p.set_psd(psd)
        return p.sigmasq()

    got = plan(True)
    if kind == "f32":
        ref = h.astype(np.complex128)
    else:
        st, s = Q.quantize_rows(h, kind)
        ref = st * s[:, None]
    # FP64 sums of n/2 positive terms in any order: n/2 x 2^-53 at most
    assert np.allclose(got, O.sigmasq(ref, w), rtol=max(1e-13, n * 2.0 ** -54), atol=0)
    assert got[-1] == 0.0
    assert np.array_equal(got, plan(False))  # the same sums from the stored rows


@pytest.mark.parametrize("lg,count,batch", [(12, 37, 1), (14, 5, 0), (20, 70, 0)])
def test_generated_rows_are_the_generators_rows(mf, lg, count, batch):
    """Blocks in the filter's scratch (or, where that holds no row, in a buffer) against rows generated alone."""
    n, fs = 1 << lg, 1024.0
    rng = np.random.default_rng(7)
    m1, m2 = rng.uniform(1.2, 20, count), rng.uniform(1.2, 20, count)
    psd = synth.psd_bins(n, fs)
    p = mf.Plan(fs, n, 1, 20.0, fs / 2, 5.0, n, max_triggers=16)
    if batch:
        p.set_batch(batch)
    p.set_psd(psd)
    p.bank_reserve(count)
    p.bank_generate_taylorf2(0, m1, m2, 20.0)
    rows = torch.zeros((count, n // 2 + 1), dtype=torch.complex64, device=DEV)
    a, b = np.ascontiguousarray(m1), np.ascontiguousarray(m2)
    assert mf.load().mf_taylorf2(a.ctypes.data, b.ctypes.data, count, fs, n, 20.0, rows.data_ptr(), n // 2 + 1,
                                 None) == mf.MF_OK
    q = mf.Plan(fs, n, 1, 20.0, fs / 2, 5.0, n, max_triggers=16)
    q.set_psd(psd)
    q.load_bank(rows)
    assert np.array_equal(p.sigmasq(), q.sigmasq())
