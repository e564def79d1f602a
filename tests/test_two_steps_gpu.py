"""Several time steps in one launch (csrc/lbm_strip.cu on large grids, two at a
time; csrc/lbm_tile.cu on small ones, four or two): the FP32 storages' step() of
several steps takes these kernels, single steps never do, and both give the same
state bit for bit -- the walls, the columns the one-step kernel updates one node
at a time, odd widths, and every place at which strips and their segments, or
the windows, can end."""
import numpy as np
import pytest

from paper_2011_15073_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu


def state_after(nx, ny, parts, field, **opts):
    with lbm.Cavity(nx, ny, 0.7, 1e-2, 1e5, 6.2, 0.6, **opts) as c:
        if field:
            c.set_darcy_field(inputs.darcy_field(1, nx, ny))
        c.set_state_f64(*inputs.perturbed_state(c.get_state_f64(), seed=nx + ny, amp=1e-2))
        for k in parts:
            c.step(k)
        host = np.empty(c.state_bytes(), np.uint8)
        c.get_state(host)
        assert lbm.debug_padding_canary(c.ctx) == 0
    # with the implicit tau the tau plane is no state
    return host[:14 * nx * ny * 4] if opts.get("tau_iters") else host


# 600,000 nodes (2,000,000 with the implicit tau) or more take the kernel; the
# widths put the right wall at every offset class of the 60-column strips and
# the 64-column tiles, the smallest and tallest grids end the segments' range
@pytest.mark.parametrize("nx,ny,opts", [
    (1024, 600, dict(prec="f32d")), (1021, 613, dict(prec="f32")), (961, 640, dict(prec="f32d", clamp_mode=1)),
    (1022, 600, dict(prec="f32")), (128, 4700, dict(prec="f32d")), (129, 4800, dict(prec="f32", clamp_mode=1)),
    (9600, 64, dict(prec="f32d")), (1500, 1400, dict(prec="f32", tau_iters=2, clamp_mode=1)),
    (1501, 1403, dict(prec="f32d", tau_iters=1))])
@pytest.mark.parametrize("field", [False, True])
def test_equals_single_steps_bit_for_bit(nx, ny, opts, field):
    one = state_after(nx, ny, [1] * 21, field, **opts)
    two = state_after(nx, ny, [7, 14], field, **opts)
    assert np.array_equal(one, two)


def test_in_replayed_graphs():
    """Graphs of double steps: lengths that are no multiple of four, and odd remainders."""
    one = state_after(1024, 600, [1] * 31, False, prec="f32d")
    for g in (2, 6, 8):
        assert np.array_equal(one, state_after(1024, 600, [11, 20], False, prec="f32d", graph_steps=g))


# at most 152 windows of 56 x 10 nodes (four steps) or 60 x 14 (two); widths and
# heights one more and one less than whole windows, the walls on the windows'
# first and last columns, the smallest width that takes the kernel
@pytest.mark.parametrize("nx,ny,opts", [
    (64, 2, dict(prec="f32d")), (65, 65, dict(prec="f32")), (112, 20, dict(prec="f32d", clamp_mode=1)),
    (113, 21, dict(prec="f32")), (111, 19, dict(prec="f32d")), (191, 64, dict(prec="f32d")),
    (256, 256, dict(prec="f32d", tau_iters=2)), (129, 301, dict(prec="f32", tau_iters=1, clamp_mode=1)),
    (300, 300, dict(prec="f32d")), (301, 281, dict(prec="f32"))])
@pytest.mark.parametrize("field", [False, True])
def test_small_grids_equal_single_steps_bit_for_bit(nx, ny, opts, field):
    one = state_after(nx, ny, [1] * 83, field, **opts)
    many = state_after(nx, ny, [7, 76], field, **opts)   # 4 + 2 + 1, and a replayed graph
    assert np.array_equal(one, many)


@pytest.mark.parametrize("opts", [dict(prec="f32d"), dict(prec="f32", clamp_mode=1), dict(prec="f32d", tau_iters=2)])
def test_batches_equal_single_steps_bit_for_bit(opts):
    """A batch large enough for two steps per launch: cavities of one strip and
    of several, of few rows and many, in one list of units."""
    grids = [(64, 16), (65, 301), (127, 130), (512, 512), (191, 77), (700, 499), (300, 300)]
    if opts.get("tau_iters"):
        grids += [(1024, 1024), (601, 603)]
    cases = [dict(nx=a, ny=b, n=0.7, Da=1e-2, Ra=1e5, Pr=6.2, porosity=0.6) for a, b in grids]
    with lbm.Batch(cases, **opts) as batch:
        for i, (nx, ny) in enumerate(grids):
            f, g, tau = lbm.get_state_f64(batch.case_ctx(i), nx, ny)
            lbm.set_state_f64(batch.case_ctx(i), *inputs.perturbed_state((f, g, tau), seed=nx + ny, amp=1e-2))
        for k in (7, 2, 12):
            batch.step(k)
        for i, (nx, ny) in enumerate(grids):
            host = np.empty(lbm.state_bytes(batch.case_ctx(i)), np.uint8)
            lbm.get_state(batch.case_ctx(i), host)
            one = state_after(nx, ny, [1] * 21, False, **opts)
            assert np.array_equal(one, host[:one.size]), (nx, ny)
