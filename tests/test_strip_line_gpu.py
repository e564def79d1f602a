"""Grids on both sides of the line from which large FP32 grids take two steps per
launch (csrc/lbm_strip.cu): the kernel that is the faster one there, and the same
bits as single steps.  The widths put the right wall at several offsets of the
strips and tiles, as tests/test_two_steps_gpu.py does."""
import numpy as np
import pytest

from paper_2011_15073_gb300 import lbm
from test_two_steps_gpu import state_after


# 657,000 nodes in tiles of 64 columns, times the tiles' columns over those of the
# strips of 60
@pytest.mark.parametrize("nx,ny,want", [
    (1024, 640, "step"), (1024, 676, "step"), (1024, 677, "strips"), (900, 640, "step"), (900, 655, "strips"),
    (256, 2800, "step"), (160, 4096, "strips"), (128, 4800, "step"), (701, 499, "step"), (840, 840, "strips"),
    (130, 3300, "strips"), (130, 3200, "step"), (30000, 30000, "strips")])
def test_the_line(nx, ny, want):
    for prec in ("f32", "f32d"):
        assert lbm.bench_steps_per_launch(nx, ny, sms=152, prec=prec)[1] == want


@pytest.mark.gpu
@pytest.mark.parametrize("nx,ny,opts", [
    (1024, 677, dict(prec="f32d")), (1021, 677, dict(prec="f32")), (961, 740, dict(prec="f32d", clamp_mode=1)),
    (1022, 677, dict(prec="f32")), (128, 7370, dict(prec="f32d")), (129, 3300, dict(prec="f32", clamp_mode=1)),
    (10950, 64, dict(prec="f32d")), (1024, 676, dict(prec="f32d")), (1021, 601, dict(prec="f32"))])
@pytest.mark.parametrize("field", [False, True])
def test_equals_single_steps_bit_for_bit(nx, ny, opts, field):
    one = state_after(nx, ny, [1] * 21, field, **opts)
    assert np.array_equal(one, state_after(nx, ny, [7, 14], field, **opts))


@pytest.mark.gpu
def test_in_replayed_graphs():
    one = state_after(1024, 677, [1] * 31, False, prec="f32d")
    for g in (2, 6, 8):
        assert np.array_equal(one, state_after(1024, 677, [11, 20], False, prec="f32d", graph_steps=g))
