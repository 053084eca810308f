"""The step below tol of the mixed solve: a right-hand side whose residual lies
between tol / 2 and tol is refined once more, and once only. Here the residual
cannot fall much below a floor: g = (closure rows of u_p) + noise of 3e-5 max |u_p|,
so that the rounding of the float64-accurate applies of K q + u_p (about 1e-15 to
1e-14 of u_p) is 1e-11 to 1e-9 of ||b||. With tol at 1.1 to 1.7 times that floor
the solve has to stay converged, with the density that its residual belongs to,
and ends after at most five steps: two to come within tol (each divides the
residual by 1e5 as long as the floor allows it), one more where rounding puts it
above tol, the further one, and one to spare; a step repeated until max_refine
takes all twelve."""
import contextlib

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layer,kappa2", [("double", 0.0), ("single", 5.0)])
@pytest.mark.parametrize("nrhs", [1, 3])
def test_one_step_below_tol(layer, kappa2, nrhs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_05507_gb300 import Context, Problem
    P = W.sphere_exp(N=32, radius=0.7)
    rng = np.random.default_rng(5)
    f = np.stack([P.f() * (1.0 + 0.3 * k) for k in range(nrhs)])
    with contextlib.closing(Context(0)) as ctx, \
            contextlib.closing(Problem(ctx, torch.from_numpy(P.phi).cuda(), P.grid.h, P.grid.origin, kappa2, layer)) as prob:
        c = prob.classification()
        t, gm, partner = c["t"], c["gm"], c["partner"]

        def closure(v):
            return t * v[gm] + (1.0 - t) * v[partner]
        up = [prob.particular(f[k], "fp64").reshape(-1) for k in range(nrhs)]
        noise = [3e-5 * np.abs(v).max() * rng.standard_normal(gm.size) for v in up]
        g = np.stack([closure(v) + e for v, e in zip(up, noise)])
        low = prob.solve_batched(f, g, tol=1e-14, precision="mixed", max_refine=12, max_iter=2000,
                                 allow_not_converged=True)[2]
        floor = max(s["rel_residual"] for s in low)
        assert 1e-11 <= floor <= 1e-8, floor
        for factor in (1.1, 1.2, 1.4, 1.7):
            tol = factor * floor
            q, u, stats = prob.solve_batched(f, g, tol=tol, precision="mixed", max_refine=12, max_iter=2000)
            for k, s in enumerate(stats):
                assert s["rel_residual"] <= tol and s["refinements"] <= 5, (factor, floor, s)
                # the residual is that of the density returned
                v = prob.potential_apply(q[k], "fp64").reshape(-1) + up[k]
                r = np.linalg.norm(g[k] - closure(v)) / np.linalg.norm(noise[k])
                assert r <= 2.0 * tol, (factor, r, tol)
                assert np.array_equal(np.asarray(u[k]).reshape(-1)[c["flags"].reshape(-1) == 0],
                                      np.zeros(int((c["flags"] == 0).sum())))
