"""The plain sweep's 4096-long columns, in both compilations (one CTA per SM up
to 152 CTAs, two beyond): every field after two sweeps against the FP64 chain,
t_2DF with its packed column among them.  Tolerance as for the other sweeps."""

import pytest

import oracle as O
from gpu_util import field, make_plan, oracle_fields, rel
from paper_1704_00865_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [32, 512, 768])
@pytest.mark.parametrize("stripes", [True, False])
def test_long_columns_match_the_chain(nx, stripes):
    from paper_1704_00865_gb300 import build, wf
    build.build()
    wf.load()
    prob = synth.make_problem(4096, nx, 37, mask_frac=0.05, stripes=stripes)
    ch = O.Chain(O.build_parts(prob, merge_2df=False, split_f=0.5, split_fp=0.25))
    plan = make_plan(prob, merge_2df=0, split_f=0.5, split_fp=0.25)
    for lam in (20.0, 1.0):
        ch.sweep(lam)
        plan.iterate(lam, 1)
    for fid, ref in oracle_fields(ch).items():
        assert rel(field(plan, fid), ref) < 2e-5, fid
    plan.close()
