"""What the server charges a job for (host only): the grid that it will create for it, without the records of
kernels that a batch lane never launches."""
import types

import pytest

from paper_1410_2817_gb300 import inputs


@pytest.mark.parametrize("n", [48, 64, 200])
def test_batched_jobs_are_not_charged_for_records(n):
    from paper_1410_2817_gb300 import build, sl
    from paper_1410_2817_gb300.serve import GpuExecutor
    build.build()
    ex = types.SimpleNamespace(sl=sl, dtype_code=GpuExecutor.dtype_code, tile_config=0)
    for wl in (inputs.workload_swirl(n), inputs.workload_burgers(n), inputs.workload_kelvin(n)):
        for max_order in {1, 2, wl.max_order}:
            wl.max_order = max_order
            planes = 2 * wl.nfields * wl.nnodes * 4

            def workspace(cfg):
                return sl.sl_grid_workspace_bytes(sl.make_desc(
                    2, wl.n, wl.nfields, sl.SL_F32, max_order=max_order, velocity=wl.velocity,
                    velocity_params=list(wl.velocity_params), tile_config=cfg))

            charged = GpuExecutor.bytes_of(ex, inputs.Job(1, 0.0, wl, "f32")) - planes
            # a batch lane's grid has no records; a lane of its own runs the default kernels
            assert charged == workspace(1 if wl.velocity == "swirl2d" else 0)
            if max_order == 2:
                assert charged == workspace(1)


@pytest.mark.parametrize("wl", [inputs.workload_burgers(64), inputs.workload_deform3d(16, steps=2)], ids=["2d", "3d"])
def test_a_job_that_fits_without_records_is_admitted(wl):
    """A budget that holds the job's grid without records, but not with them: the job goes without."""
    from paper_1410_2817_gb300 import build, sl
    from paper_1410_2817_gb300.serve import GpuExecutor, Scheduler, job_grid
    build.build()
    job = inputs.Job(1, 0.0, wl, "f32")
    with_records, without = job_grid(sl, job, 0)[1], job_grid(sl, job, 1)[1]
    assert without < with_records
    for budget, cfg in ((with_records, 0), (with_records - 1, 1), (without, 1)):
        ex = types.SimpleNamespace(sl=sl, dtype_code=GpuExecutor.dtype_code, tile_config=0, budget=budget)
        sch = Scheduler(budget, bytes_of=lambda j: GpuExecutor.bytes_of(ex, j))
        assert not sch.submit(job).rejected and len(sch.admit(0.0)) == 1
        assert job_grid(sl, job, 0, budget)[0] == cfg
    assert Scheduler(without - 1, bytes_of=lambda j: without).submit(job).rejected
