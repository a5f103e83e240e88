"""GPU parity of the Welch estimate over segment counts: one, two and three segments, counts on both sides of the
shared-memory steps of the median, the largest, and rows of equal values."""

import numpy as np
import pytest

from oracle import mf_oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def mf(lib):
    from paper_2309_00019_gb300 import mf as m
    return m


@pytest.mark.parametrize("average", ["mean", "median"])
@pytest.mark.parametrize("segments,stride", [(1, 4096), (2, 4096), (3, 1000), (190, 64), (193, 64), (4096, 16)])
def test_welch_over_segment_counts(mf, segments, stride, average):
    fs, seg = 1024.0, 4096
    rng = np.random.default_rng(segments)
    x = rng.standard_normal((3, seg + (segments - 1) * stride + 7)).astype(np.float32)
    x[2] = 0.0
    got = mf.psd_welch(torch.from_numpy(x).to(DEV), fs, seg, stride, average).cpu().numpy()
    ref = O.psd_welch(x.astype(np.float64), fs, seg, stride, average)
    assert not got[2].any()
    # white data: every bin has power of the FP32 transform's own scale (relative accuracy as in the other tests of
    # the estimate, of the typical bin where a single periodogram can be near zero)
    assert np.abs(got[:2] - ref[:2]).max() <= 1e-4 * np.median(ref[:2])
