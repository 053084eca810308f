"""Boundary operator and solves at N = 256 for bodies of few planes, whose applies
run on kernels that thicker bodies do not reach: the even-odd schedule on the whole
grid (whole rows, and split frequencies) and on the window of 192 nodes, the
direct i pass at 192 and 256 planes' length, and the double-float i pass of at most
128 planes. Each precision, by the library's choice and as five passes, against the
float64 potential of the whole grid, which transforms every plane: float64 and
double-float to 1e-12 and float32 to 2e-6 of the largest potential, the bounds of
the oracle comparisons of the same applies. A batched solve equals its single ones
to the bit."""
import contextlib

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

N = 256
TOL = {"fp32": 2e-6, "fp64": 1e-12, "df64": 1e-12}


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_05507_gb300 import Context, set_conv_schedule
    c = Context(0)
    yield c
    set_conv_schedule("auto")
    c.close()


def body(axes, centre, kappa2=3.0):
    """Ellipsoid with semi-axes and centre in grid steps (centre from the middle of the grid)."""
    h = 2.0 / N
    return W._make(f"flat_N{N}", W.cell_centred(N),
                   lambda x, y, z: ((x - centre[0] * h) / (axes[0] * h)) ** 2 + ((y - centre[1] * h) / (axes[1] * h)) ** 2
                   + ((z - centre[2] * h) / (axes[2] * h)) ** 2 - 1.0,
                   kappa2, "double", lambda x, y, z: W.sol_exp_sum(x, y, z, kappa2))


# semi-axis a along z: about 2 a + 3 source planes (an odd count where the centre
# is half a step off); the first four fit the window of 192 nodes
BODIES = [((90.0, 90.0, 10.0), (20.0, -30.0, 90.5)), ((91.0, 80.0, 45.0), (0.0, 0.0, 0.0)),
          ((90.0, 85.0, 45.9), (0.0, 30.0, -70.0)), ((85.0, 90.0, 55.0), (0.5, 0.0, 60.5)),
          ((105.0, 60.0, 6.0), (0.0, 10.0, -100.0)), ((105.0, 90.0, 30.0), (10.0, 0.0, 0.5)),
          ((105.0, 90.0, 39.0), (-15.0, 0.0, 40.0)), ((110.0, 100.0, 51.0), (0.0, 0.0, 0.5)),
          ((105.0, 100.0, 62.0), (0.0, 10.0, 30.0)), ((105.0, 100.0, 69.5), (0.0, 0.0, -20.0))]


@pytest.mark.parametrize("axes,centre", BODIES)
@pytest.mark.parametrize("layer", ["double", "single"])
def test_apply_matches_whole_grid(ctx, axes, centre, layer):
    import torch
    from paper_2502_05507_gb300 import Problem, set_conv_schedule
    P = body(axes, centre)
    with contextlib.closing(Problem(ctx, torch.from_numpy(P.phi).cuda(), P.grid.h, P.grid.origin, P.kappa2, layer)) as prob:
        cl = prob.classification()
        q = torch.from_numpy(W.random_density(prob.n_unknowns, seed=72)).cuda()
        v = prob.potential_apply(q, "fp64").reshape(-1).cpu().numpy()
        ref = cl["t"] * v[cl["gm"]] + (1.0 - cl["t"]) * v[cl["partner"]]
        big = np.max(np.abs(v))
        for schedule in ("auto", "passes", "persist"):
            set_conv_schedule(schedule)
            for precision in ("fp32", "df64", "fp64"):
                a = prob.boundary_apply(q, precision).cpu().numpy()
                assert np.max(np.abs(a - ref)) <= TOL[precision] * big, (schedule, precision)
        set_conv_schedule("auto")


@pytest.mark.parametrize("axes,centre", [BODIES[1], BODIES[6], BODIES[8]])
def test_batch_equals_single(ctx, axes, centre):
    import torch
    from paper_2502_05507_gb300 import Problem
    P = body(axes, centre)
    with contextlib.closing(Problem(ctx, torch.from_numpy(P.phi).cuda(), P.grid.h, P.grid.origin, P.kappa2, "double")) as prob:
        g0 = P.g_at(prob.boundary_points())
        f0 = torch.from_numpy(P.f()).cuda()
        f = torch.stack([f0, 0.5 * f0])
        g = torch.from_numpy(np.stack([g0, 1.5 * g0])).cuda()
        u = prob.solve_batched(f, g, tol=1e-9, precision="mixed")[1]
        for k in range(2):
            one = prob.solve_batched(f[k:k + 1], g[k:k + 1], tol=1e-9, precision="mixed")[1]
            assert torch.equal(one[0], u[k])
        m = torch.from_numpy(P.phi < 0).cuda()
        exact = torch.from_numpy(P.u_exact()).cuda()
        assert float((u[0] - exact)[m].abs().max() / exact[m].abs().max()) <= 1e-4
