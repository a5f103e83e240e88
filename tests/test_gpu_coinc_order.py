"""GPU checks of the order of the coincidence records on every way they are put in order: short lists, long ones, far more
(template, shift) bins than records, a bin too crowded to count ranks in, and no device memory for the ordering (the
allocation is refused by a stand-in for cudaMalloc, in a process of its own)."""

import os
import subprocess
import sys

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KEYS = ("tmpl", "shift", "sample0", "sample1")


def make(mf, tmpl, sel, shift, shifts, rho, max_coincs=1 << 20):
    n, fs, f_low = 1 << 14, 512.0, 30.0
    rng = np.random.default_rng(tmpl)
    bank = np.stack([synth.taylorf2(n, fs, 2.0 + 0.01 * i, 1.5, f_low) for i in range(tmpl)]).astype(np.complex64)
    p = mf.Plan(fs, n, 2, f_low, fs / 2, 2.5, 64)
    p.set_psd(synth.psd_bins(n, fs))
    p.load_bank(torch.from_numpy(bank).to(DEV))
    d = torch.from_numpy(np.stack([synth.coloured_noise_fd(rng, n, fs) for _ in range(2)]).astype(np.complex64)).to(DEV)
    s = None if sel is None else torch.tensor(sel, dtype=torch.int32, device=DEV)
    p.filter(d, subset=s)
    p.coincide(torch.zeros(tmpl, dtype=torch.int32, device=DEV), shift, shifts, 8, rho, max_coincs=max_coincs)
    return p


def in_order(co):
    return np.array_equal(co, co[np.lexsort([co[k] for k in reversed(KEYS)])])


# (template count, copies of template 0 in the selection, shift, shifts, rho_c, records at least, at most)
@pytest.mark.parametrize("tmpl,copies,shift,shifts,rho,least,most", [
    (40, 0, 500, 1, 4.8, 100, 2047),           # short: on the host
    (200, 0, 500, 20, 4.5, 2048, 1 << 20),     # on the device
    (3, 0, 3, 1500000, 6.0, 20000, 1 << 20),   # 4.5 million bins, in proportion to the records
    (3, 0, 3, 1500000, 6.2, 2048, 19000),      # and not: on the host
    (1, 12000, 1, 0, 4.5, 65537, 1 << 20),     # one bin: too crowded
    (1, 2000, 1, 0, 4.5, 2048, 65536),         # one bin, ranks counted
])
def test_records_in_order(lib, tmpl, copies, shift, shifts, rho, least, most):
    from paper_2309_00019_gb300 import mf
    p = make(mf, tmpl, [0] * copies if copies else None, shift, shifts, rho)
    co, found, _ = p.coincs()
    assert least <= found <= most and len(co) == found
    assert in_order(co)
    if copies:  # the same records that often
        one = make(mf, tmpl, [0], shift, shifts, rho).coincs()[0]
        assert len(one) * copies == found and np.array_equal(co[::copies], one)
    few = p.coincs(cap=7)[0]
    assert np.array_equal(few, co[:7])


SHIM = """
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static size_t limit = (size_t)-1;
static int refused = 0;
void shim_limit(size_t n) { limit = n; }
int shim_refused(void) { return refused; }
int cudaMalloc(void** p, size_t n) {
  static int (*real)(void**, size_t) = 0;
  if (!real) real = (int (*)(void**, size_t))dlsym(dlopen("libcudart.so.13", RTLD_LAZY), "cudaMalloc");
  if (n > limit) {
    ++refused;
    *p = 0;
    return 2; /* cudaErrorMemoryAllocation */
  }
  return real(p, n);
}
"""

CHILD = """
import ctypes, os, sys
sys.path[:0] = [{root!r}, {tests!r}]
import numpy as np
import torch
from paper_2309_00019_gb300 import mf
from test_gpu_coinc_order import make, in_order
shim = ctypes.CDLL({so!r})
p = make(mf, 200, None, 500, 20, 4.5)
torch.cuda.synchronize()
shim.shim_limit(ctypes.c_size_t(4096))
a, found, st = p.coincs()
refused = shim.shim_refused()
shim.shim_limit(ctypes.c_size_t(2 ** 64 - 1))
b, _, _ = p.coincs()
assert refused >= 1 and shim.shim_refused() == refused, refused
assert st == mf.MF_OK and found == len(a) >= 2048 and in_order(a) and np.array_equal(a, b)
print("ok")
"""


def test_no_memory_for_the_ordering(lib, tmp_path):
    src, so = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so), str(src), "-ldl"], check=True)
    child = CHILD.format(root=ROOT, tests=os.path.join(ROOT, "tests"), so=str(so))
    r = subprocess.run([sys.executable, "-c", child], env={**os.environ, "LD_PRELOAD": str(so)}, capture_output=True,
                       text=True, timeout=180)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
