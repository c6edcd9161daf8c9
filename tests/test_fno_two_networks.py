"""Networks alive at the same time.  Networks of one channel group run the same
compiled kernels, and what the runtime keeps per kernel (its limit on dynamic
shared memory) outlives the creation that set it: a network made later, with a
smaller footprint, must leave the earlier one working, bit for bit."""

import numpy as np
import pytest

import fake_gpu

# (n, width, mx, my) of the first and of the second network, one channel group
# each: fewer modes, fewer channels, a larger map (whose rows take less)
PAIRS = [((64, 8, 16, 8), (64, 8, 4, 4)), ((64, 16, 16, 8), (64, 10, 4, 4)), ((64, 32, 32, 8), (64, 32, 16, 8)),
         ((256, 32, 16, 16), (256, 24, 8, 8)), ((64, 32, 16, 16), (256, 32, 16, 16)), ((64, 64, 32, 8), (64, 40, 8, 8))]


def test_launches_of_the_first_network_are_taken_after_a_second_one(tmp_path):
    # the network's launches against the runtime's rule, without a GPU
    fake_gpu.run(tmp_path, f"""
    bad = []
    for pair in {PAIRS!r}:
        nets = [(s[0], wf.FNO(s[0], 1, synth.fno_init(1, *s[1:], 2), width=s[1], mx=s[2], my=s[3], layers=2,
                              stream=NO_STREAM)) for s in pair]
        for n, net in nets + nets[:1]:
            x, t, y = (C.c_void_p(fake.fake_alloc(4 * k * n * n)) for k in (2, 1, 1))
            loss = C.c_double()
            first = fake.fake_launches()
            rc = [lib.wf_fno_forward(net.h, x, y, 1), lib.wf_fno_gradient(net.h, x, t, 1, None, C.byref(loss)),
                  lib.wf_fno_train_step(net.h, x, t, 1, 1e-3, C.byref(loss))]
            assert len(launches(first)) > 20
            if rc != [wf.WF_OK] * 3 or any(l[3] for l in launches(first)):
                bad.append((pair, n, rc, [l for l in launches(first) if l[3]]))
    assert not bad, bad
    """)


@pytest.mark.gpu
@pytest.mark.parametrize("a,b", PAIRS)
def test_the_first_network_gives_the_same_after_a_second_one(a, b):
    import torch
    from gpu_util import dev
    from paper_1704_00865_gb300 import build, synth, wf
    build.build()
    wf.load()

    def net(n, width, mx, my):
        return wf.FNO(n, 1, synth.fno_init(5, width, mx, my, 2), width=width, mx=mx, my=my, layers=2)

    n = a[0]
    rng = np.random.default_rng(n)
    x, t = dev(rng.standard_normal((1, 2, n, n)).astype(np.float32)), dev(rng.standard_normal((1, n, n)).astype(np.float32))
    first = net(*a)
    y0, y1 = torch.empty(1, n, n, device="cuda"), torch.empty(1, n, n, device="cuda")
    first.forward(x, y0, 1)
    loss0, g0 = first.gradient(x, t, 1)
    second = net(*b)
    first.forward(x, y1, 1)
    loss1, g1 = first.gradient(x, t, 1)
    second.close()
    first.close()
    assert torch.equal(y0, y1) and loss0 == loss1 and np.array_equal(g0, g1)
