"""The i pass as a direct sum over the planes (pruned applies of few planes)
against the FFT i pass: boundary_apply, which transforms only the planes that
hold sources, equals the closure rows of potential_apply, which transforms
every plane (more than the direct sum takes at N >= 64). Slabs from the
thinnest the geometry allows to the most planes the direct sum takes, odd and
even plane counts, off-centre, both layers; float64 and double-float to 1e-12
and float32 to 2e-6 of the largest potential, the bounds of the oracle
comparisons of the same applies."""
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


def slab(N, half, z0, kappa2):
    """A disk (semi-axes 0.75, 0.6) of half thickness `half` grid steps centred `z0` steps off the middle."""
    h = 2.0 / N
    return W._make(f"slab_N{N}", W.cell_centred(N),
                   lambda x, y, z: (x / 0.75) ** 2 + (y / 0.6) ** 2 + ((z - z0 * h) / (half * h)) ** 2 - 1.0,
                   kappa2, "double", lambda x, y, z: W.sol_exp_sum(x, y, z, kappa2))


# (N, half thickness, offset): 7 to 9 planes, then odd and even counts up to the direct sum's most
SLABS = [(64, 1.2, 0.3), (64, 9.4, 3.0), (64, 18.3, -2.2), (64, 23.9, 0.5), (128, 1.2, 20.5), (128, 14.6, -7.5),
         (128, 29.9, 0.5), (128, 30.4, 1.0), (128, 38.9, 0.0)]


@pytest.mark.parametrize("schedule", ["passes", "auto"])
@pytest.mark.parametrize("precision", ["fp32", "df64", "fp64"])
@pytest.mark.parametrize("layer", ["double", "single"])
@pytest.mark.parametrize("N,half,z0", SLABS)
def test_direct_sum_matches_fft(ctx, N, half, z0, layer, precision, schedule):
    import torch
    from paper_2502_05507_gb300 import Problem, set_conv_schedule
    P = slab(N, half, z0, 5.0)
    with contextlib.closing(Problem(ctx, torch.from_numpy(P.phi).cuda(), P.grid.h, P.grid.origin, P.kappa2, layer)) as prob:
        ax, lo, hi = prob.conv_planes()
        cl = prob.classification()
        q = torch.from_numpy(W.random_density(prob.n_unknowns, seed=61)).cuda()
        set_conv_schedule("passes")
        v = prob.potential_apply(q, "fp64").cpu().numpy().reshape(-1)
        ref = cl["t"] * v[cl["gm"]] + (1.0 - cl["t"]) * v[cl["partner"]]
        set_conv_schedule(schedule)
        Aq = prob.boundary_apply(q, precision).cpu().numpy()
        assert np.max(np.abs(Aq - ref)) <= TOL[precision] * np.max(np.abs(v)), (ax, lo, hi)
