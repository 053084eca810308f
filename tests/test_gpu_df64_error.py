"""Error of the double-float boundary operator (single layer, whose values do not
cancel; relative L2 norm, mean over six densities) against the float64 potential of
the whole grid, which is within 2e-15. Bounds: a tenth above the errors of the same
operators made of transforms of powers of two along every axis, over the whole grid.

- The direct sum over the planes ("passes", whole grid): 4.55e-15 and 5.09e-15 with
  the transform; with sums that are not put in order after every block of rows
  5.43e-15 and 6.11e-15.
- The window of 3/4 of the grid: 4.06e-15, 4.03e-15, 4.20e-15, 4.58e-15 and 5.69e-15
  with the whole grid's transforms; where the sums of the window's lengths are not put
  in order, 5.38e-15 to 6.69e-15."""
import contextlib

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def body(N, axes):
    """Ellipsoid with semi-axes in half-widths of the grid, off its middle."""
    return W._make(f"body_N{N}", W.cell_centred(N),
                   lambda x, y, z: ((x - 0.4 / N) / axes[0]) ** 2 + ((y + 0.3 / N) / axes[1]) ** 2
                   + ((z - 0.2 / N) / axes[2]) ** 2 - 1.0,
                   0.0, "single", lambda x, y, z: W.sol_exp_sum(x, y, z, 0.0))


CASES = [(128, (0.85, 0.5, 0.35), "passes", 4.55e-15), (256, (0.85, 0.6, 0.33), "passes", 5.09e-15),
         (64, (0.7, 0.5, 0.15), "auto", 4.06e-15), (64, (0.6, 0.6, 0.6), "auto", 4.03e-15),
         (128, (0.7, 0.5, 0.15), "auto", 4.20e-15), (128, (0.6, 0.6, 0.6), "auto", 4.58e-15),
         (256, (0.7, 0.65, 0.33), "auto", 5.69e-15)]


@pytest.mark.parametrize("N,axes,schedule,before", CASES)
def test_operator_error(N, axes, schedule, before):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_05507_gb300 import Context, Problem, set_conv_schedule
    P = body(N, axes)
    err = []
    with contextlib.closing(Context(0)) as ctx, \
            contextlib.closing(Problem(ctx, torch.from_numpy(P.phi).cuda(), P.grid.h, P.grid.origin, 0.0, "single")) as prob:
        c = prob.classification()
        try:
            for seed in range(6):
                q = torch.from_numpy(W.random_density(prob.n_unknowns, seed=seed)).cuda()
                set_conv_schedule("passes")
                v = prob.potential_apply(q, "fp64").reshape(-1).cpu().numpy()
                ref = c["t"] * v[c["gm"]] + (1.0 - c["t"]) * v[c["partner"]]
                set_conv_schedule(schedule)
                a = prob.boundary_apply(q, "df64").cpu().numpy()
                err.append(np.linalg.norm(a - ref) / np.linalg.norm(ref))
        finally:
            set_conv_schedule("auto")
    assert np.mean(err) <= 1.1 * before, err
