"""What the passes ask for to spread their CTAs over the SMs, and the residual's
kernels with them, on a runtime without a GPU (fake_cudart.cpp).  Up to 57 KB of
shared memory (of an SM's 228) leave room for a second and third CTA."""

import fake_gpu


def test_column_pass_leaves_room_for_two_row_ctas(tmp_path):
    fake_gpu.run(tmp_path, """
    def column_pass(ny, nx, **kw):
        p = synth.make_problem(ny, nx, 1)
        plan = wf.Plan(ny, nx, 7, wf.make_params(autotune=0, **kw), stream=NO_STREAM)
        plan.set_problem(p.d, p.pixel_var, p.mask, p.C, p.P1f, p.Pst, p.stripe_amp2)
        at = fake.fake_launches()
        plan.iterate(1.0, 1)
        plan.close()
        smem, = {l[2] for l in launches(at) if "col_pass" in l[1]}
        return smem

    # 128 column CTAs, 256 row CTAs (two an SM): not spread
    assert column_pass(256, 1024) <= 57 * 1024
    # 128 column CTAs, 384, 512 and 1024 row CTAs: one to an SM
    for ny in (384, 512, 1024):
        assert column_pass(ny, 1024) > 113 * 1024, ny
    """)


def test_residual_kernels_take_the_spread_passes_split_on_middle_sized_maps(tmp_path):
    fake_gpu.run(tmp_path, """
    def splits(ny, nx):
        p = synth.make_problem(ny, nx, 1)
        plan = wf.Plan(ny, nx, 7, wf.make_params(autotune=0), stream=NO_STREAM)
        plan.set_problem(p.d, p.pixel_var, p.mask, p.C, p.P1f, p.Pst, p.stripe_amp2)
        at = fake.fake_launches()
        plan.residual()
        plan.close()
        names = [l[1] for l in launches(at)]
        out = {fake.fake_carveout(at + i) for i, n in enumerate(names) if "row_kernel" in n or "col_kernel" in n}
        assert len(names) == 5  # four of the residual and the controller
        return out

    for shape in ((512, 1024), (1024, 128), (128, 1024)):
        assert splits(*shape) == {100}, shape
    for shape in ((64, 64), (128, 128), (1024, 1024), (2048, 512)):
        assert splits(*shape) == {-1}, shape
    """)
