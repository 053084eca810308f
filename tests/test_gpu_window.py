"""Pruned applies on a window of 3/4 of the grid (transforms of length 3N/2,
where the sources fit it along every axis) against the whole grid: the
boundary operator by the library's own choice equals the closure rows of
potential_apply, which transforms every node. Bodies that fill the window to
the node, that miss it by one node along one axis (whole grid), off-centre
against every face of the grid, flat ones (swapped axes) and wide ones (the
five passes), every layer; float64 and double-float to 1e-12 and float32 to
2e-6 of the largest potential, the bounds of the oracle comparisons of the
same applies. Solves agree with the whole grid's to 1e-9."""
import contextlib

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

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


def body(N, axes, centre, kappa2=3.0):
    """Ellipsoid with semi-axes and centre in grid steps (centre from the middle of the grid)."""
    h = 2.0 / N
    return W._make(f"body_N{N}", W.cell_centred(N),
                   lambda x, y, z: ((x - centre[0] * h) / (axes[0] * h)) ** 2 + ((y - centre[1] * h) / (axes[1] * h)) ** 2
                   + ((z - centre[2] * h) / (axes[2] * h)) ** 2 - 1.0,
                   kappa2, "double", lambda x, y, z: W.sol_exp_sum(x, y, z, kappa2))


def _problem(ctx, P, layer):
    import torch
    from paper_2502_05507_gb300 import Problem
    return Problem(ctx, torch.from_numpy(P.phi).cuda(), P.grid.h, P.grid.origin, P.kappa2, layer)


# the window has 3 N / 4 nodes; a semi-axis a gives about 2 a + 4 source planes
BODIES = [(32, (9.9, 8.0, 6.0), (3.0, -2.5, 0.0)), (32, (9.6, 4.0, 9.5), (-4.0, 0.0, 3.5)),
          (32, (11.4, 11.0, 9.0), (0.0, 0.0, 0.0)), (64, (21.9, 21.8, 5.0), (-7.0, 0.5, -20.0)),
          (64, (22.9, 15.0, 21.0), (0.5, 9.0, 0.0)), (128, (45.9, 30.0, 10.0), (0.0, 5.0, -40.0)),
          (128, (45.6, 45.4, 45.2), (15.0, -15.0, 14.5)), (128, (46.0, 20.0, 46.0), (-14.0, 30.0, 14.0)),
          (128, (48.4, 20.0, 12.0), (0.5, 0.0, 0.0)), (256, (93.0, 90.0, 70.0), (30.0, -33.0, 10.0)),
          (256, (94.0, 93.9, 93.5), (0.0, 0.5, 31.0))]


@pytest.mark.parametrize("precision", ["fp32", "df64", "fp64"])
@pytest.mark.parametrize("layer", ["double", "single", "direct"])
@pytest.mark.parametrize("N,axes,centre", BODIES)
def test_window_apply_matches_whole_grid(ctx, N, axes, centre, layer, precision):
    import torch
    from paper_2502_05507_gb300 import set_conv_schedule
    P = body(N, axes, centre)
    with contextlib.closing(_problem(ctx, P, layer)) as prob:
        cl = prob.classification()
        qh = W.random_density(prob.n_unknowns, seed=71)
        q = torch.from_numpy(qh).cuda()
        set_conv_schedule("passes")   # the whole grid
        v = prob.potential_apply(q, "fp64").cpu().numpy().reshape(-1)
        if layer == "direct":
            number = np.zeros(N ** 3, np.int64)
            gp = prob.gamma_plus()
            number[gp] = np.arange(gp.size) + prob.n_gm
            ref = np.concatenate([cl["t"] * qh[: prob.n_gm] + (1.0 - cl["t"]) * qh[number[cl["partner"]]],
                                  qh[prob.n_gm:] - v[gp]])
        else:
            ref = cl["t"] * v[cl["gm"]] + (1.0 - cl["t"]) * v[cl["partner"]]
        set_conv_schedule("auto")
        Aq = prob.boundary_apply(q, precision).cpu().numpy()
        assert np.max(np.abs(Aq - ref)) <= TOL[precision] * max(np.max(np.abs(v)), np.max(np.abs(ref)))


@pytest.mark.parametrize("N,axes,centre,nrhs", [(128, (45.0, 40.0, 12.0), (3.0, 0.0, 0.0), 3), (128, (46.0, 45.0, 44.0), (0.0, -14.0, 0.0), 1)])
def test_window_solve_matches_whole_grid(ctx, N, axes, centre, nrhs):
    import torch
    from paper_2502_05507_gb300 import set_conv_schedule
    P = body(N, axes, centre)
    with contextlib.closing(_problem(ctx, P, "double")) as prob:
        g = P.g_at(prob.boundary_points())
        f = torch.from_numpy(np.stack([P.f() * (1.0 + 0.2 * k) for k in range(nrhs)])).cuda()
        gg = torch.from_numpy(np.stack([g * (1.0 - 0.1 * k) for k in range(nrhs)])).cuda()
        out = {}
        for schedule in ("passes", "auto"):
            set_conv_schedule(schedule)
            out[schedule] = prob.solve_batched(f, gg, tol=1e-11, precision="mixed")[1].cpu().numpy()
        a, b = out["auto"], out["passes"]
        assert np.max(np.abs(a - b)) <= 1e-9 * np.max(np.abs(b))
