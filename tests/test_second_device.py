"""One process, two GPUs: what the library sets for a kernel (its limit on
dynamic shared memory) is kept by the runtime per kernel and device, so every
launch must be taken on a device that another one was used before.  On a
runtime without a GPU (fake_cudart.cpp), which holds each launch to that rule."""

import fake_gpu


def test_every_launch_is_taken_on_a_second_device(tmp_path):
    fake_gpu.run(tmp_path, """
    def problem(ny, nx):
        p = synth.make_problem(ny, nx, 1)
        return p.d, p.pixel_var, p.mask, p.C, p.P1f, p.Pst, p.stripe_amp2

    sizes = [(32, 32), (512, 384), (1024, 1024), (1536, 768), (2048, 512), (64, 4096), (4096, 128)]
    inputs = [problem(*s) for s in sizes]
    for dev in (0, 1):
        fake.fake_set_device(dev)
        at = fake.fake_launches()
        # the transforms, with and without a plan, at every column length
        for ny in (32, 64, 128, 256, 384, 512, 768, 1024, 1536, 2048, 4096):
            nx = 64
            x, y = (C.c_void_p(fake.fake_alloc(4 * ny * nx)) for _ in range(2))
            for inverse in (0, 1):
                assert lib.wf_fft2_noalloc(ny, nx, x, y, inverse, None) == wf.WF_OK, (dev, ny, inverse)
            plan = wf.Plan(ny, nx, wf.WF_PART_WHITE, stream=NO_STREAM)
            for inverse in (0, 1):
                assert lib.wf_fft2(plan.h, x, y, inverse, 0) == wf.WF_OK, (dev, ny, inverse)
            plan.close()
        # sweeps (both shapes, merged and plain; the one-launch form), residual and fields
        for (ny, nx), inp in zip(sizes, inputs):
            for kw in (dict(autotune=0), dict(autotune=2), dict(merge_2df=0, split_f=0.5, split_fp=0.0)) + (
                    (dict(sweep_kernel=1),) if ny == nx == 1024 else ()):
                plan = wf.Plan(ny, nx, 7, wf.make_params(**kw), stream=NO_STREAM)
                plan.set_problem(*inp)
                plan.iterate(1.0, 2)
                plan.residual()
                plan.get_field(wf.WF_FIELD_S, np.empty((ny, nx), np.float32))
                plan.close()
        here = launches(at)
        assert len(here) > 100 and all(l[0] == dev for l in here) and not any(l[3] for l in here)
    """)
