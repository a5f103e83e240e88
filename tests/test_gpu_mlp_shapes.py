"""GPU checks of the ranking network's products at the edges of their tiles (odd sizes, one row, K below one step and
across several, rows that need padding) against the FP64 oracle, and of the ranking against the network's own logits."""

import numpy as np
import pytest

from oracle import mlp_oracle as M

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def mfmod(lib):
    from paper_2309_00019_gb300 import mf
    return mf


@pytest.mark.parametrize("dims,B", [((3, 20, 2, 37), 13), ((1, 8, 1, 9), 1), ((9, 65, 3, 33), 65), ((5, 64, 1, 64), 64),
                                    ((16, 72, 2, 321), 130)])
def test_products_over_shapes(mfmod, dims, B):
    rng = np.random.default_rng(sum(dims) + B)
    net = mfmod.MLP(*dims, max_batch=B + 3)
    theta = M.init_params(rng, dims).astype(np.float32)
    net.set_params(theta)
    x = rng.standard_normal((B, dims[0])).astype(np.float32)
    nv = rng.integers(1, dims[3] + 1, B).astype(np.int32)
    nv[0] = dims[3]
    lab = np.array([rng.integers(0, v) for v in nv], np.int32)
    xd, nvd = torch.from_numpy(x).to(DEV), torch.from_numpy(nv).to(DEV)
    logits = torch.full((B, dims[3]), np.nan, device=DEV)
    net.forward(xd, logits)
    ref, _ = M.forward(theta.astype(np.float64), x, dims)
    got = logits.cpu().numpy()
    # BF16 operands (2^-9 each) through at most four layers: as for the network's own sizes
    assert np.linalg.norm(got - ref) <= 2e-2 * np.linalg.norm(ref)
    loss, grad = torch.zeros(1, device=DEV), torch.full((net.n_params,), np.nan, device=DEV)
    net.loss_grad(xd, nvd, torch.from_numpy(lab).to(DEV), loss, grad)
    rl, rg = M.loss_and_grad(theta.astype(np.float64), x, nv, lab, dims)
    g = grad.cpu().numpy().astype(np.float64)
    assert float(loss.item()) == pytest.approx(rl, rel=2e-2)
    assert np.linalg.norm(g - rg) <= 3e-2 * np.linalg.norm(rg)
    # the ranking is that of the logits: best first, ties to the lower slot, -1 after the last valid slot
    k = min(64, dims[3])
    out, cnt = torch.zeros((B, k), dtype=torch.int32, device=DEV), torch.zeros(B, dtype=torch.int32, device=DEV)
    net.topk(xd, nvd, k, out, count=cnt)
    out, cnt = out.cpu().numpy(), cnt.cpu().numpy()
    for i in range(B):
        want = np.argsort(-got[i, : nv[i]], kind="stable")[:k]
        assert cnt[i] == len(want) and np.array_equal(out[i, : len(want)], want) and (out[i, len(want):] == -1).all()
