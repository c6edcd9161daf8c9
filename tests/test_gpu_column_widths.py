"""The column kernels of the transforms, the residual and the export of s at
long columns, on both sides of the rule for narrow CTAs (no more of them than
SMs): transforms against numpy, s and the residual of a swept state against the
FP64 chain.  Tolerances: those of the tests at other sizes (transforms 2e-6,
fields 2e-5, residual terms 2e-3: g = S^-1 s in FP32 at high k)."""

import numpy as np
import pytest

import oracle as O
from gpu_util import field, make_plan, pack_spectrum, rel, unpack_spectrum
from paper_1704_00865_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(1536, 512), (1536, 768), (2048, 512), (2048, 768), (4096, 256), (4096, 384)]


@pytest.fixture(scope="module")
def wf():
    from paper_1704_00865_gb300 import build, wf
    build.build()
    wf.load()
    return wf


@pytest.mark.parametrize("ny,nx", SHAPES)
def test_transforms(wf, ny, nx):
    x = np.random.default_rng(ny + nx).standard_normal((ny, nx)).astype(np.float32)
    plan = wf.Plan(ny, nx, wf.WF_PART_WHITE)
    X = np.fft.rfft2(x.astype(np.float64))
    assert rel(unpack_spectrum(plan.fft2(x), ny, nx), X) < 2e-6
    assert rel(plan.fft2(pack_spectrum(X), inverse=True).reshape(ny, nx), x) < 2e-6
    plan.close()


@pytest.mark.parametrize("merge", [1, 0])
@pytest.mark.parametrize("ny,nx", SHAPES)
def test_export_and_residual(wf, ny, nx, merge):
    prob = synth.make_problem(ny, nx, 51, mask_frac=0.05)
    P = O.build_parts(prob, merge_2df=bool(merge), split_f=0.5, split_fp=0.5 * merge)
    ch = O.Chain(P)
    plan = make_plan(prob, merge_2df=merge, split_f=0.5, split_fp=0.5 * merge)
    for lam in (20.0, 1.0):
        ch.sweep(lam)
        plan.iterate(lam, 1)
    assert rel(field(plan, wf.WF_FIELD_S), ch.s) < 2e-5
    u, m = plan.residual()
    plan.close()
    rho, gm, g = O.residual_terms(P, ch.s)
    du = np.where(P.unmasked, P.d, 0.0)
    assert u == pytest.approx(np.linalg.norm(rho) / np.linalg.norm(du), rel=2e-3)
    assert m == pytest.approx(np.linalg.norm(gm) / np.linalg.norm(g), rel=2e-3)
