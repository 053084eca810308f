"""Point sets formed from words of 32 nodes, bit for bit against the oracle, where
the words have edges: lines shorter than a word (N = 8, 16), nodes on both sides
of a word's end, and sets without structure (random signs)."""
import contextlib

import numpy as np
import pytest

from oracle import grid as OG

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,density", [(8, 0.5), (8, 0.1), (16, 0.5), (32, 0.3), (64, 0.5), (128, 0.02)])
def test_random_sets_match_the_oracle(N, density):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_05507_gb300 import Context, Problem
    rng = np.random.default_rng(N)
    phi = rng.uniform(0.1, 1.0, (N, N, N))
    inner = (slice(2, N - 2),) * 3   # M+ and gamma- off the faces of the box
    phi[inner][rng.random((N - 4,) * 3) < density] *= -1.0
    phi[rng.random(phi.shape) < 0.02] = 0.0   # zero is outside M+
    h = 2.0 / N
    ref = OG.classify(phi, h, -1.0)
    with contextlib.closing(Context(0)) as ctx, \
            contextlib.closing(Problem(ctx, torch.from_numpy(phi).cuda(), h, -1.0, 0.0, "double")) as prob:
        c = prob.classification()
        xs = prob.boundary_points()
    fl = c["flags"]
    assert np.array_equal(fl & 1 != 0, ref.inside)
    assert np.array_equal(fl & 2 != 0, ref.gm)
    assert np.array_equal(fl & 4 != 0, ref.gp)
    assert np.array_equal(fl & 8 != 0, ref.dnode)
    assert np.array_equal((fl >> 4).astype(np.int64) * ref.gm, ref.count * ref.gm)
    assert np.array_equal(c["gm"], ref.gm_idx)
    assert np.array_equal(c["partner"], ref.partner)
    assert np.array_equal(c["t"], ref.t)
    assert np.array_equal(xs, ref.xstar)
