"""Both compiled shapes of the row and the column pass at every row length and
every column length, on square and ragged maps, for each kind of sweep: with
stripes (merged and plain), with 1/f only, white only.  Every field after two
sweeps against the FP64 chain.

Tolerance: that of the other sweep tests, 2e-5 -- FP32 transforms of a few 1e-7
each, eight per two sweeps, and updates whose weights stay below 1.
"""

import numpy as np
import pytest

import oracle as O
from gpu_util import field, make_plan, oracle_fields, rel
from paper_1704_00865_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(32, 32), (128, 64), (32, 128), (64, 256), (256, 384), (384, 768), (768, 1536), (1536, 512), (512, 1024),
          (1024, 2048), (2048, 64), (32, 4096), (4096, 32)]
KINDS = {"merged": dict(), "plain": dict(merge=0), "no_stripes": dict(stripes=False),
         "white": dict(stripes=False, one_over_f=False)}


@pytest.fixture(scope="module")
def wf():
    from paper_1704_00865_gb300 import build, wf
    build.build()
    wf.load()
    return wf


@pytest.mark.parametrize("kind", list(KINDS))
@pytest.mark.parametrize("shape", SHAPES)
def test_both_shapes_match_the_chain(wf, shape, kind):
    kw = dict(KINDS[kind])
    merge = kw.pop("merge", 1)
    prob = synth.make_problem(*shape, 31, mask_frac=0.05, stripe_rows_vary=kw.get("stripes", True), **kw)
    split_fp = 0.5 if merge else 0.25
    P = O.build_parts(prob, merge_2df=bool(merge), split_f=0.5, split_fp=split_fp)
    ch = O.Chain(P)
    for lam in (20.0, 1.0):
        ch.sweep(lam)
    refs = oracle_fields(ch)
    seen = set()
    for autotune in (0, 2):
        plan = make_plan(prob, merge_2df=merge, split_f=0.5, split_fp=split_fp, autotune=autotune)
        for lam in (20.0, 1.0):
            plan.iterate(lam, 1)
        for fid, ref in refs.items():
            assert rel(field(plan, fid), ref) < 2e-5, (plan.shapes(), fid)
        seen.add(plan.shapes())
        plan.close()
    assert len(seen) == 2  # the row pass has two shapes at every length


@pytest.mark.parametrize("shape", [(64, 64), (256, 384), (1024, 512), (2048, 64), (4096, 32)])
def test_one_correction_with_its_source_matches_the_chain(wf, shape):
    # The column pass with the masked-pixel source, staged and not, in the CTA
    # of the packed column and in the others: twenty sweeps, then a correction
    # of two sweeps (its data the residual on unmasked pixels, its source
    # S^-1 s on masked ones), against the same steps in FP64.  Tolerance 1e-3:
    # that of the residual's own tests (g = S^-1 s in FP32 at high k), which
    # bounds the correction's error relative to s.
    import dataclasses
    import torch
    from gpu_util import dev
    prob = synth.make_problem(*shape, 33, mask_frac=0.05)
    plan = wf.Plan(*shape, wf.parts_of(prob), wf.make_params(residual_every=2, max_iters=20, refine=1,
                                                             refine_max_iters=2))
    out = torch.empty(*shape, device="cuda")
    plan.solve(*[dev(a) for a in (prob.d, prob.pixel_var, prob.mask, prob.C, prob.P1f, prob.Pst, prob.stripe_amp2)],
               wf.make_schedule("fixed", [1.0], [0]), 0.0, out=out)
    plan.close()
    P = O.build_parts(prob, merge_2df=True, split_f=0.5, split_fp=0.5)
    ch = O.Chain(P)
    for _ in range(20):
        ch.sweep(1.0)
    rho, j, _ = O.residual_terms(P, ch.s)
    J, N0 = O.to_basis("2DF", j), P.parts[0].N
    co = O.Chain(dataclasses.replace(P, d=rho))
    T1 = co.T(1, 1.0)
    for _ in range(2):
        co.sweep(1.0)
        Y = O.to_basis("2DF", co.t[1])
        co.dd[0] = O.from_basis("2DF", ((P.C + N0) * Y + T1 * P.C * J) / (P.C + N0 + T1))
        co.s = O.from_basis("2DF", P.C * (Y + (N0 + T1) * J) / (P.C + N0 + T1))
    ref = ch.s - co.s
    assert rel(out.cpu().numpy(), ref) < 1e-3
