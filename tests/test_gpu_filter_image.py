"""GPU checks of the FP16 column pass at the edges of its launch (fewer columns than warps, one column each, several
rounds, one to three detectors, every bank type, odd selections) against the FP32 intermediate."""

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


@pytest.mark.parametrize("dets,tmpl,sel,kind,inter", [
    (1, 1, None, "f32", "f16"), (1, 2, [1], "f16", "f16x2"), (2, 3, None, "bf16", "f16"), (3, 5, [0, 1, 2, 4], "f32", "f16x2"),
    (1, 9, [2, 3, 5, 8], "f16", "f16"), (2, 4, None, "bf16", "f16x2"),
])
def test_images_agree_with_the_fp32_intermediate(mf, dets, tmpl, sel, kind, inter):
    n, fs, f_low, window, thr = 1 << 20, 2048.0, 30.0, 1 << 15, 4.5
    rng = np.random.default_rng(tmpl + dets)
    dtype = {"f32": mf.MF_F32, "f16": mf.MF_F16, "bf16": mf.MF_BF16}[kind]
    m1, m2 = rng.uniform(1.4, 9.0, tmpl), rng.uniform(1.4, 9.0, tmpl)
    rows = synth.taylorf2_torch(n, fs, m1, m2, f_low, DEV)
    d = np.stack([synth.coloured_noise_fd(rng, n, fs) for _ in range(dets)])
    amp = 9.0 / synth.taylorf2_norm_continuum(m1[-1], m2[-1], f_low, fs / 2)
    d += synth.taylorf2(n, fs, m1[-1], m2[-1], f_low, t0=200.0, amp=amp)
    data = torch.from_numpy(d.astype(np.complex64)).to(DEV)
    sub = None if sel is None else torch.tensor(sel, dtype=torch.int32, device=DEV)
    p = mf.Plan(fs, n, dets, f_low, fs / 2, thr, window, dtype=dtype, max_triggers=1 << 16)
    p.set_psd(synth.psd_bins(n, fs))
    p.bank_reserve(tmpl, dtype)
    p.bank_set_rows(0, rows) if kind == "f32" else p.bank_quantize_rows(0, rows)
    out = {}
    for im in ("f32", inter):
        p.set_intermediate({"f32": mf.MF_F32, "f16": mf.MF_F16, "f16x2": mf.MF_F16X2}[im])
        p.filter(data, subset=sub)
        t = p.triggers()[0]
        out[im] = {(int(x["det"]), int(x["tmpl"]), int(x["sample"]) // window): x for x in t}
    a, b = out["f32"], out[inter]
    tol = 1e-3 if inter == "f16" else 1e-4  # the stated accuracy of the two intermediates
    for k in set(a) ^ set(b):
        assert abs(float(a.get(k, b.get(k))["snr"]) / thr - 1) <= tol, k
    assert len(set(a) & set(b)) >= dets
    for k in set(a) & set(b):
        assert abs(float(a[k]["snr"]) / float(b[k]["snr"]) - 1) <= tol, k
        if float(a[k]["snr"]) > 7:
            assert a[k]["sample"] == b[k]["sample"]
