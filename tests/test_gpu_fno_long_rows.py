"""The network's row transform with one group of warps per block (four blocks per
SM and more): sums of half a row, 256 and 512 terms, against the FP64 oracle.
Tolerance as for the other network tests, 2e-5 (FP32 sums of up to 512 terms)."""

import numpy as np
import pytest

from oracle import fno_oracle as F
from gpu_util import dev, rel
from test_gpu_fno import _net, wf  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


# maps x channels x blocks of 64 rows: 768 blocks each, 608 are four per SM
@pytest.mark.parametrize("n,nb,width,mx,my", [(512, 3, 32, 16, 8), (1024, 1, 48, 16, 4), (1024, 1, 48, 32, 4)])
def test_forward_with_one_group_per_block(wf, n, nb, width, mx, my):  # noqa: F811
    import torch
    net, p = _net(wf, n, nb, width, mx, my, 1)
    x = np.random.default_rng(n + mx).standard_normal((nb, 2, n, n)).astype(np.float32)
    y = torch.empty(nb, n, n, device="cuda")
    net.forward(dev(x), y, nb)
    net.close()
    assert rel(y.cpu().numpy(), F.forward(p, x.astype(np.float64))) < 2e-5
