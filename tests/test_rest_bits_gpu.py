"""Runs from rest with FP32 deviations: ahead of the flow the deviations are
subnormal, and their rounding too may not depend on how many steps a launch
takes, nor on whether a cavity runs in a batch (csrc/lbm_device.cuh, vscale)."""
import numpy as np
import pytest

from paper_2011_15073_gb300 import lbm

pytestmark = pytest.mark.gpu


# sizes that take four, two (window), one, and two (strips) steps per launch, wide
# enough that what comes from the side walls, a column per step, is subnormal by then
@pytest.mark.parametrize("nx,ny,opts", [
    (1200, 40, dict(tau_iters=0)), (1100, 90, dict(tau_iters=0)), (1201, 37, dict(tau_iters=2)), (700, 400, dict(tau_iters=2)),
    (1024, 700, dict(tau_iters=0)), (1500, 1400, dict(tau_iters=2)), (1501, 1403, dict(tau_iters=1))])
@pytest.mark.parametrize("n", [1.0, 0.6])
def test_runs_from_rest_have_the_same_bits(nx, ny, opts, n):
    params = dict(n=n, Da=1e-2, Ra=1e5, Pr=6.2, porosity=0.6)
    opts = dict(prec="f32d", clamp_mode=1, **opts)
    host = []
    k = 300
    for parts in ([1] * k, [k]):
        with lbm.Cavity(nx, ny, **params, **opts) as c:
            for m in parts:
                c.step(m)
            host.append(np.empty(c.state_bytes(), np.uint8))
            c.get_state(host[-1])
    with lbm.Batch([dict(nx=nx, ny=ny, **params)] * 2, **opts) as b:
        b.step(k)
        host.append(np.empty(lbm.state_bytes(b.case_ctx(1)), np.uint8))
        lbm.get_state(b.case_ctx(1), host[-1])
    size = 14 * nx * ny * 4 if opts["tau_iters"] else host[0].size   # with the implicit tau the tau plane is no state
    values = host[0][:14 * nx * ny * 4].view(np.float32)
    assert ((values != 0) & (np.abs(values) < 2.0 ** -126)).any()   # there are subnormal ones
    for h in host[1:]:
        assert np.array_equal(host[0][:size], h[:size])
