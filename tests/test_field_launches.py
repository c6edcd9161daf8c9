"""Kernels that reading a field takes: one per transform it needs, and one to
bring a column-tiled field without a column transform to rows.  Counted on a
runtime without a GPU (fake_cudart.cpp)."""

import fake_gpu


def test_each_field_takes_one_kernel_per_step(tmp_path):
    fake_gpu.run(tmp_path, """
    for ny, nx in ((32, 64), (2048, 32), (384, 96 * 8)):
        for merge in (1, 0):
            p = synth.make_problem(ny, nx, 1)
            plan = wf.Plan(ny, nx, 7, wf.make_params(merge_2df=merge, split_f=0.5, split_fp=0.5 * merge),
                           stream=NO_STREAM)
            plan.set_problem(p.d, p.pixel_var, p.mask, p.C, p.P1f, p.Pst, p.stripe_amp2)
            # s from the messenger next to it, t_2DF through a column transform;
            # t_RF and d_2DF untiled; d_RF as it is; then the rows
            want = {wf.WF_FIELD_S: 2, wf.WF_FIELD_T_RF: 2, wf.WF_FIELD_D_2DF: 2, wf.WF_FIELD_D_RF: 1}
            if not merge:
                want[wf.WF_FIELD_T_2DF] = 2
            for f, n in want.items():
                n0, l0 = plan.launch_count(), fake.fake_launches()
                plan.get_field(f, np.empty((ny, nx), np.float32))
                assert plan.launch_count() - n0 == fake.fake_launches() - l0 == n, (ny, nx, merge, f)
            plan.close()
    """)
