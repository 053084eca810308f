"""Values that take each way through the conversion of float64 inputs to the
float32 and double-float applies (normal, zero, and so small that the parts are
not normal float32 numbers): the particular solution is linear in f, so that of
f times a power of two is that of f times the same power. double-float to 1e-12,
float32 to 2e-6 of the largest value, the bounds of the same applies against the
oracle."""
import contextlib

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 2e-6, "df64": 1e-12}


@pytest.mark.parametrize("precision", ["fp32", "df64"])
@pytest.mark.parametrize("power", [40, -20, -56, -62, -66])
def test_scaled_inputs(precision, power):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_05507_gb300 import Context, Problem
    p = W.sphere_exp(N=32, radius=0.7)
    rng = np.random.default_rng(11)
    f = rng.standard_normal(p.phi.shape)
    f[rng.random(f.shape) < 0.1] = 0.0
    f[rng.random(f.shape) < 0.1] = -0.0
    f[rng.random(f.shape) < 0.1] = 1e-310
    with contextlib.closing(Context(0)) as ctx, \
            contextlib.closing(Problem(ctx, torch.from_numpy(p.phi).cuda(), p.grid.h, p.grid.origin, 1.0, "double")) as prob:
        one = prob.particular(f, precision)
        far = np.ldexp(prob.particular(np.ldexp(f, power), precision), -power)
        ref = prob.particular(f, "fp64")
    big = np.abs(ref).max()
    assert np.abs(one - ref).max() <= TOL[precision] * big
    assert np.abs(far - ref).max() <= TOL[precision] * big
