"""GPU check of the Welch median on both sides of each number of keys that a lane holds: 1,024, 2,048 and 4,096 segments,
random and many equal values, against a sort of the same periodograms taken one segment at a time."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("segments", [512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 3001, 4095, 4096])
def test_medians_are_the_middle_values(lib, segments):
    from paper_2309_00019_gb300 import mf
    fs, seg = 512.0, 4096
    rng = np.random.default_rng(segments)
    # twelve kinds of segment, each many times (ties around the middle), in any order, without overlap
    kinds = rng.standard_normal((12, seg)).astype(np.float32)
    order = rng.integers(0, 12, (2, segments))
    x = torch.from_numpy(kinds).to(DEV)[torch.from_numpy(order).to(DEV)].reshape(2, segments * seg).contiguous()
    got = mf.psd_welch(x, fs, seg, seg, "median").cpu().numpy()
    one = np.stack([mf.psd_welch(torch.from_numpy(k[None]).to(DEV), fs, seg, seg, "median").cpu().numpy()[0] for k in kinds])
    i = np.arange(1, (segments - 1) // 2 + 1)
    bias = 1.0 + np.sum(1.0 / (2.0 * i + 1.0) - 1.0 / (2.0 * i))
    for d in range(2):
        v = np.sort(one[order[d]], axis=0)
        ref = 0.5 * (v[(segments - 1) // 2] + v[segments // 2]) / bias
        assert np.allclose(got[d], ref, rtol=1e-13, atol=0)  # the same values; the bias is a sum of some thousand terms
