"""The rule by which lbm_step takes several steps per launch
(lbm_bench_steps_per_launch; csrc/lbm_tile.cu, csrc/lbm_strip.cu): one wave of
windows on the SMs that the GPU has.  No GPU needed: the SM count is given."""
import pytest

from paper_2011_15073_gb300 import lbm


# windows of four steps bring 56 x 10 nodes forward, of two 60 x 14
@pytest.mark.parametrize("nx,ny,sms,want", [
    (256, 256, 152, (4, "tile")),    # 5 x 26 = 130 windows
    (256, 256, 130, (4, "tile")),
    (256, 256, 129, (2, "tile")),    # 5 x 19 = 95
    (256, 256, 95, (2, "tile")),
    (256, 256, 94, (1, "step")),
    (300, 300, 152, (2, "tile")),    # 6 x 30, 5 x 22
    (384, 384, 152, (1, "step")),
    (63, 40, 152, (1, "step")),
    (64, 2, 1, (1, "step")),         # two windows' columns
    (56 * 2, 10, 2, (4, "tile")),
])
def test_windows_fill_one_wave_of_the_gpu(nx, ny, sms, want):
    for prec in ("f32", "f32d"):
        assert lbm.bench_steps_per_launch(nx, ny, sms=sms, prec=prec) == want
    for other in (dict(prec="f64"), dict(prec="f16s"), dict(prec="f32d", layout=1), dict(prec="f32d", staging=1)):
        assert lbm.bench_steps_per_launch(nx, ny, sms=sms, **other) == (1, "step")


def test_large_grids_take_strips():
    assert lbm.bench_steps_per_launch(4096, 4096, sms=152, prec="f32d") == (2, "strips")
    assert lbm.bench_steps_per_launch(2048, 2048, sms=152, prec="f32", tau_iters=2) == (2, "strips")
    for other in (dict(prec="f64"), dict(prec="f16d"), dict(prec="f32", layout=1), dict(prec="f32", staging=1)):
        assert lbm.bench_steps_per_launch(4096, 4096, sms=152, **other) == (1, "step")
    for nx, ny in ((127, 20000), (20000, 63)):   # narrower or lower than the strips take
        assert lbm.bench_steps_per_launch(nx, ny, sms=152, prec="f32d")[1] != "strips"


def test_bad_arguments():
    for nx, ny, sms in ((1, 64, 152), (64, 1, 152), (64, 64, -1)):
        with pytest.raises(lbm.LBMError):
            lbm.bench_steps_per_launch(nx, ny, sms=sms, prec="f32")
