"""What the fixed-point collision of the FP64 storage admits
(csrc/lbm_collide_fixed.cuh): every state it takes is computed as in wider
arithmetic, every other one is left to the FP64 collision.  On the host over the
whole range (tests/host/fixed_range_check.cu), on the GPU with dense fluids."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("flags", [["-O2"], ["-O1", "-Xcompiler", "-fsanitize=signed-integer-overflow,"
                                             "-fno-sanitize-recover=signed-integer-overflow", "-lubsan"]],
                         ids=["plain", "overflow-checked"])
def test_admitted_states_are_right_and_refused_ones_unchanged(tmp_path, flags):
    """The tests of a node's ranges look at sums that may wrap, which signed
    integers may not: checked too."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "fixed_range_check")
    src = os.path.join(ROOT, "tests", "host", "fixed_range_check.cu")
    inc = os.path.join(ROOT, "paper_2011_15073_gb300", "csrc")
    subprocess.run([nvcc, "-std=c++17", "-I", inc, src, "-o", exe, *flags], check=True, timeout=300)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.startswith("OK"), (r.stdout + r.stderr)[-2000:]


# f and g to 1e-12, as every FP64 run against the oracle.  tau: 1e-14 in the
# populations (8 steps of some ten roundings) is 1e-12 in the strain rate, over
# that of gamma_1, 0.01 U_c / L = 8.2e-6, times |n - 1| = 0.3: below 1e-7 relative
@pytest.mark.gpu
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("density", [0.45, 1.3, 1.4, 1.75, 1.85, 1.95])
def test_dense_fluids_equal_the_oracle(density, layout):
    import oracle
    from paper_2011_15073_gb300 import inputs, lbm
    nx, ny = 70, 33
    params = dict(n=0.7, Da=1e-2, Ra=1e5, Pr=6.2, porosity=0.6, clamp_mode=1)
    ref = oracle.Cavity.from_params(nx, ny, **params)
    f, g, tau = inputs.perturbed_state(ref.get_state(), seed=3)
    f = f * density * (1.0 + 0.05 * np.random.default_rng(5).uniform(-1, 1, (ny, nx)))
    ref.set_state(f, g, tau)
    ref.step(8)
    with lbm.Cavity(nx, ny, prec="f64", layout=layout, **params) as cav:
        cav.set_state_f64(f, g, tau)
        cav.step(8)
        got = cav.get_state_f64()
    want = ref.get_state()
    for a, b, tol in zip(got, want, (1e-12, 1e-12, 1e-7 * want[2])):
        assert (np.abs(a - b) <= tol).all()


@pytest.mark.gpu
def test_nodes_beyond_the_drag_limit_pay_for_one_collision_only():
    """Where the Darcy drag is above the fixed-point collision's limit at every
    node (a small Darcy number), the step costs what it costs where no node
    tries it (n = 2, which its parameters exclude): both run the same FP64
    arithmetic, one after a test that fails at once.  Shortest of ten runs of 20
    steps each, in turn; with the limit tested after most of the fixed-point
    work it was 6 % more."""
    import torch
    from paper_2011_15073_gb300 import lbm
    best = {}
    stream = torch.cuda.Stream()
    runs = {n: lbm.Cavity(512, 512, n, 1e-7, 1e5, 6.2, 0.6, prec="f64", clamp_mode=1, cuda_stream=stream) for n in (1.9, 2.0)}
    for _ in range(10):
        for n, cav in runs.items():
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            cav.step(2)
            a.record(stream)
            cav.step(20)
            b.record(stream)
            b.synchronize()
            best[n] = min(best.get(n, 1e9), a.elapsed_time(b))
    for n, cav in runs.items():
        lat = cav.lattice()
        tau = cav.get_state_f64()[2]
        assert np.isfinite(tau).all() and (lat.eps / lat.K * (tau - 0.5) / 3 > 1).all()
        cav.close()
    assert best[1.9] < 1.03 * best[2.0], best
