"""Device memory of the ranking network: per layer and row one FP32 pre-activation and one BF16 activation, and a few
buffers that do not grow with the depth."""

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_memory_per_layer(lib):
    from paper_2309_00019_gb300 import mf

    width, depth, batch = 1024, 12, 8192
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net = mf.MLP(8, width, depth, 64, max_batch=batch)
    used = free - torch.cuda.mem_get_info()[0]
    # parameters, gradient and two moments in FP32, a BF16 copy; 6 bytes per layer and activation; 10 for the backward
    # pass; a tenth for the small buffers and the allocator's steps of 2 MB
    need = 18 * net.n_params + (6 * depth + 10) * batch * width
    assert used <= 1.1 * need, (used, need)
    net.close()
