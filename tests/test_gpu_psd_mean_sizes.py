"""GPU check of the Welch mean on both sides of the number of segments from which on more warps share a bin, against the
means of the same periodograms taken one segment at a time."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("segments", [31, 4096, 4097, 4129, 9000])
def test_means_are_those_of_the_segments(lib, segments):
    from paper_2309_00019_gb300 import mf
    fs, seg = 512.0, 4096
    rng = np.random.default_rng(segments)
    kinds = rng.standard_normal((12, seg)).astype(np.float32)
    order = rng.integers(0, 12, (2, segments))
    x = torch.from_numpy(kinds).to(DEV)[torch.from_numpy(order).to(DEV)].reshape(2, segments * seg).contiguous()
    got = mf.psd_welch(x, fs, seg, seg, "mean").cpu().numpy()
    one = np.stack([mf.psd_welch(torch.from_numpy(k[None]).to(DEV), fs, seg, seg, "mean").cpu().numpy()[0] for k in kinds])
    for d in range(2):
        ref = (np.bincount(order[d], minlength=12)[:, None] * one).sum(0) / segments
        # FP64 sums of positive terms in any order: n 2^-53 at most
        assert np.allclose(got[d], ref, rtol=segments * 2.0 ** -53 + 1e-15, atol=0)
