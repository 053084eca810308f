"""The forms of the LGF spectrum that a problem keeps: the octant of its grid, and one
form per element type for the window of its pruned applies.

- Device memory that a further kappa^2 h^2 takes at N = 256: 20 257^3 bytes (340 MB) for
  the octants and at most 20 * 192 * 193 * 196 (145 MB) for the window; 2 MB per array
  for the granularity of allocations, and 30 MB for the rest of a problem's footprint.
- Problems of one (N, kappa^2 h^2) that need different forms share a cache in either
  order: a flat body (mixed forms), one of many planes (octants) and one that no window
  takes; then a forced schedule, which runs on the whole grid, and a solve that
  captures its steps as the first call under it. Bounds as in the tests of the same
  applies against the whole grid."""
import contextlib

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 2e-6, "fp64": 1e-12, "df64": 1e-12}


@pytest.fixture
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_05507_gb300 import Context, set_conv_schedule
    c = Context(0)
    yield c
    set_conv_schedule("auto")
    c.close()


def body(N, axes):
    """Ellipsoid with semi-axes in grid steps."""
    h = 2.0 / N
    return W._make(f"body_N{N}", W.cell_centred(N),
                   lambda x, y, z: (x / (axes[0] * h)) ** 2 + (y / (axes[1] * h)) ** 2 + (z / (axes[2] * h)) ** 2 - 1.0,
                   3.0, "double", lambda x, y, z: W.sol_exp_sum(x, y, z, 3.0))


def _problem(ctx, P, kappa2=3.0):
    import torch
    from paper_2502_05507_gb300 import Problem
    return Problem(ctx, torch.from_numpy(P.phi).cuda(), P.grid.h, P.grid.origin, kappa2, "double")


def _check_apply(prob, q, precisions):
    cl = prob.classification()
    v = prob.potential_apply(q, "fp64").reshape(-1).cpu().numpy()
    ref = cl["t"] * v[cl["gm"]] + (1.0 - cl["t"]) * v[cl["partner"]]
    for precision in precisions:
        a = prob.boundary_apply(q, precision).cpu().numpy()
        assert np.max(np.abs(a - ref)) <= TOL[precision] * np.max(np.abs(v)), precision


def test_memory_of_a_further_kappa2(ctx):
    import torch
    P = body(256, (90.0, 90.0, 30.0))
    free = []
    for kappa2 in (1.0, 2.0, 3.0):
        _problem(ctx, P, kappa2).close()
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    assert free[1] - free[2] <= 20 * 257 ** 3 + 20 * 192 * 193 * 196 + (7 * 2 + 30) * 2 ** 20


@pytest.mark.parametrize("N", [64, 128])
@pytest.mark.parametrize("order", [(0, 1, 2), (2, 1, 0), (1, 0, 2)])
def test_shared_cache(ctx, N, order):
    import torch
    from paper_2502_05507_gb300 import set_conv_schedule
    u = N / 64
    bodies = [body(N, a) for a in ((22.0 * u, 20.0 * u, 4.0 * u), (22.0 * u, 21.5 * u, 21.0 * u), (28.0 * u, 20.0 * u, 6.0 * u))]
    with contextlib.ExitStack() as stack:
        probs = [stack.enter_context(contextlib.closing(_problem(ctx, bodies[k]))) for k in order]
        qs = [torch.from_numpy(W.random_density(p.n_unknowns, seed=7)).cuda() for p in probs]
        for p, q in zip(probs, qs):
            _check_apply(p, q, ("fp32", "df64", "fp64"))
        first = [p.boundary_apply(q, "fp32") for p, q in zip(probs, qs)]
        g = [torch.from_numpy(bodies[k].g_at(p.boundary_points())).cuda() for k, p in zip(order, probs)]
        f = [torch.from_numpy(bodies[k].f()).cuda() for k in order]
        ref = [p.solve(a, b, tol=1e-10, precision="mixed")[1] for p, a, b in zip(probs, f, g)]
        set_conv_schedule("passes")
        for p, a, b, r in zip(probs, f, g, ref):
            u1 = p.solve(a, b, tol=1e-10, precision="mixed", use_graphs=True)[1]
            assert float((u1 - r).abs().max()) <= 1e-8 * float(r.abs().max())
        for p, q in zip(probs, qs):
            _check_apply(p, q, ("fp32", "df64", "fp64"))
        set_conv_schedule("auto")   # the same forms as before: the same passes, to the bit
        for p, q, a in zip(probs, qs, first):
            assert torch.equal(p.boundary_apply(q, "fp32"), a)
