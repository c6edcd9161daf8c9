"""The warm-start network's tiled kernels at the edges of their tiles -- channel
counts that do not fill a group, odd mode counts, rows shorter and longer
than a tile, fewer maps than the plan holds -- against the FP64 oracle.

Tolerances: as for the other network tests, 2e-5 for the output (FP32 sums of
up to 512 terms per layer, a few 1e-7 expected) and 2e-3 for the gradient
against central finite differences (whose own error dominates).
"""

import numpy as np
import pytest

from oracle import fno_oracle as F
from gpu_util import dev, rel
from test_gpu_fno import _net, wf  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# n, maps held, maps used, width, mx, my, layers
SHAPES = [(16, 3, 2, 2, 1, 1, 1), (16, 2, 2, 64, 8, 8, 2), (32, 2, 1, 18, 16, 16, 2), (64, 1, 1, 10, 5, 3, 3),
          (128, 2, 2, 34, 7, 9, 2), (256, 1, 1, 16, 13, 5, 1), (512, 1, 1, 32, 16, 16, 1), (1024, 1, 1, 8, 32, 32, 1)]


@pytest.mark.parametrize("n,batch,nb,width,mx,my,layers", SHAPES)
def test_forward_at_tile_edges(wf, n, batch, nb, width, mx, my, layers):  # noqa: F811
    import torch
    net, p = _net(wf, n, batch, width, mx, my, layers)
    x = np.random.default_rng(n + width).standard_normal((nb, 2, n, n)).astype(np.float32)
    # an input and an output that start 4 bytes off a 16-byte boundary
    xd = torch.empty(x.size + 1, device="cuda")[1:].view(nb, 2, n, n)
    xd.copy_(torch.from_numpy(x))
    y = torch.full((nb * n * n + 2,), 7.0, device="cuda")
    net.forward(xd, y[1:-1], nb)
    net.close()
    got = y.cpu().numpy()
    assert got[0] == 7.0 and got[-1] == 7.0
    assert rel(got[1:-1].reshape(nb, n, n), F.forward(p, x.astype(np.float64))) < 2e-5


@pytest.mark.parametrize("n,batch,nb,width,mx,my,layers", [s for s in SHAPES if s[0] <= 128])
def test_gradient_at_tile_edges(wf, n, batch, nb, width, mx, my, layers):  # noqa: F811
    net, p = _net(wf, n, batch, width, mx, my, layers, seed=3)
    rng = np.random.default_rng(n)
    x = rng.standard_normal((nb, 2, n, n)).astype(np.float32)
    t = rng.standard_normal((nb, n, n)).astype(np.float32)
    loss, g = net.gradient(dev(x), dev(t), nb)
    again = net.gradient(dev(x), dev(t), nb)[1]
    net.close()
    assert np.array_equal(g, again)
    x, t = x.astype(np.float64), t.astype(np.float64)
    assert loss == pytest.approx(F.loss(p, x, t), rel=1e-5)
    sizes = [width * 2, width] + layers * [width * width, width, width * width * 2 * my * mx * 2] + [width, 1]
    assert sum(sizes) == g.size
    o = 0
    for size in sizes:
        idx = sorted(set([o, o + size - 1] + list(range(o, o + size, max(1, size // 5)))))
        fd = F.fd_gradient(p, x, t, idx)
        assert np.linalg.norm(g[idx] - fd) <= 2e-3 * max(np.linalg.norm(fd), 1e-30), (o, size)
        o += size
