"""wf_fft2_noalloc makes its twiddle tables on the device, one entry a thread:
every length in both directions against wf_fft2, whose tables are the host's.
Tolerance: that of the transform's other comparison with wf_fft2, 5e-6 (tables
that differ by the rounding of a sine in double)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIDES = (32, 64, 128, 256, 384, 512, 768, 1024, 1536, 2048, 4096)


@pytest.mark.parametrize("n", SIDES)
@pytest.mark.parametrize("other", [32, 256])
def test_every_length_matches_the_plan(n, other):
    import torch
    from paper_1704_00865_gb300 import build, wf
    build.build()
    wf.load()
    for ny, nx in {(n, other), (other, n)}:
        x = torch.randn(ny, nx, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
        plan = wf.Plan(ny, nx, wf.WF_PART_WHITE)
        out = torch.empty_like(x)
        for inverse in (False, True):
            ref = plan.fft2(x, inverse=inverse, out=torch.empty_like(x))
            wf.wf_fft2_noalloc(ny, nx, x, out, inverse=inverse)
            torch.cuda.synchronize()
            a, b = out.cpu().numpy().astype(np.float64), ref.cpu().numpy().astype(np.float64)
            assert np.linalg.norm(a - b) <= 5e-6 * np.linalg.norm(b), (ny, nx, inverse)
        plan.close()
