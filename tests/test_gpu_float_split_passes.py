"""The conversion of float64 inputs in the five passes and the plane-fused kernels
(by integer operations, also for float32; the even-odd schedule, which takes these
sizes by itself, has the conversion instruction there): the particular solution of f
times a power of two is that of f times the same power, for values whose float32
parts are normal numbers, zeros, and below. float32 to 2e-6 and double-float to 1e-12
of the largest value, the bounds of the same applies against the oracle."""
import contextlib

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 2e-6, "df64": 1e-12}


@pytest.mark.parametrize("N,schedule", [(32, "passes"), (32, "plane"), (64, "plane"), (128, "passes_alt"), (128, "plane")])
@pytest.mark.parametrize("precision", ["fp32", "df64"])
def test_scaled_inputs(N, schedule, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_05507_gb300 import Context, Problem, set_conv_schedule
    p = W.sphere_exp(N=N, radius=0.7)
    rng = np.random.default_rng(11)
    f = rng.standard_normal(p.phi.shape)
    f[rng.random(f.shape) < 0.1] = 0.0
    f[rng.random(f.shape) < 0.1] = -0.0
    f[rng.random(f.shape) < 0.1] = 1e-310
    with contextlib.closing(Context(0)) as ctx, \
            contextlib.closing(Problem(ctx, torch.from_numpy(p.phi).cuda(), p.grid.h, p.grid.origin, 1.0, "double")) as prob:
        ref = prob.particular(f, "fp64")
        big = np.abs(ref).max()
        try:
            set_conv_schedule(schedule)
            for power in (0, 40, -20, -56, -62, -66):
                v = np.ldexp(prob.particular(np.ldexp(f, power), precision), -power)
                assert np.abs(v - ref).max() <= TOL[precision] * big, power
        finally:
            set_conv_schedule("auto")
