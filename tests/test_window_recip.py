"""CPU check of the window reciprocal that the filter kernels divide by: exact for every window at the ends of every
window and for every sample of odd ones."""

import numpy as np


def recip(w):
    return ((1 << 40) + w - 1) // w


def test_quotients_are_exact():
    n_max = 1 << 20
    rng = np.random.default_rng(0)
    windows = np.unique(np.concatenate([np.arange(1, 600), 2 ** np.arange(21), n_max - np.arange(50),
                                        rng.integers(1, n_max + 1, 300)]))
    for w in windows.tolist():
        ends = np.arange(0, n_max, w, dtype=np.uint64)
        n = np.unique(np.concatenate([ends, ends[1:] - np.uint64(1), rng.integers(0, n_max, 200).astype(np.uint64)]))
        assert int(n.max()) * recip(w) < 1 << 64
        assert np.array_equal((n * np.uint64(recip(w))) >> np.uint64(40), n // np.uint64(w)), w
