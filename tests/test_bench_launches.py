"""bench.py describes the launches that the library makes, at every size (CPU
part: the SM count is given)."""
import bench


def test_launches_follow_the_library():
    # two steps per launch on large FP32 grids, four or two on small ones, one between and otherwise
    for N, prec, want, label in ((4096, "f32d", 2, "strip_kernel (two steps per launch)"),
                                 (256, "f32d", 4, "tile_kernel (four steps per launch)"),
                                 (300, "f32", 2, "tile_kernel (two steps per launch)"),
                                 (512, "f32d", 1, "step2_kernel"), (256, "f64", 1, "step_kernel"),
                                 (4096, "f16s", 1, "step4_kernel"), (256, "f16s", 1, "step2_kernel")):
        assert bench.steps_per_launch(prec, 0, 0, 0, N, sms=152)[0] == want
        assert bench.launch_label(prec, 0, 0, 0, N, sms=152) == label
    assert bench.steps_per_launch("f32d", 1, 0, 0, 256, sms=152)[0] == 1
    assert [bench.launches_of(k, 4) for k in (0, 1, 2, 3, 4, 7, 1000)] == [0, 1, 1, 2, 1, 3, 250]
    assert [bench.launches_of(k, 2) for k in (1, 2, 7, 1000)] == [1, 1, 4, 500]
    assert bench.launches_of(1000, 1) == 1000


def test_recorded_figures_depend_on_every_step_kernel():
    assert {"lbm_tile.cu", "lbm_strip.cuh", "lbm_step.cuh", "lbm_collide_fixed.cuh"} <= set(bench.RECORD_SOURCES)
