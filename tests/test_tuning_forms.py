"""The pair of pass shapes is chosen once per map shape and process and holds
for a plan of its own and for a batch's plans alike, so the choice must not
depend on which of them came first: both time the passes as a plan of its own
launches them.  On a runtime without a GPU (fake_cudart.cpp): every pass launch
of a plan's tuning, with the shared memory it asks for, is among those of a
batch that tunes."""

import fake_gpu


def test_a_batch_tunes_the_launches_of_a_plan_of_its_own(tmp_path):
    seen = []
    for body in ("""
    plan = wf.Plan(ny, nx, 7, wf.make_params(max_iters=10), stream=NO_STREAM)
    plan.set_problem(*prob)
    """, """
    b = wf.Batch([(ny, nx)] * 2, params=wf.make_params(max_iters=10), lanes=2, stream=NO_STREAM)
    outs = [np.empty((ny, nx), np.float32) for _ in range(2)]
    b.solve([prob] * 2, wf.make_schedule("fixed", [1.0], [10]), 0.0, outs)
    """):
        out = tmp_path / f"launches{len(seen)}"
        fake_gpu.run(tmp_path, f"""
    ny = nx = 512
    p = synth.make_problem(ny, nx, 1)
    prob = (p.d, p.pixel_var, p.mask, p.C, p.P1f, p.Pst, p.stripe_amp2)
    {body}
    open({str(out)!r}, "w").write("\\n".join(sorted({{f"{{n}} {{s}}" for _, n, s, _ in launches() if "_pass_kernel" in n}})))
    """)
        seen.append(set(out.read_text().split("\n")))
    assert len(seen[0]) == 4  # two shapes of each pass
    assert seen[0] <= seen[1], seen[0] - seen[1]
