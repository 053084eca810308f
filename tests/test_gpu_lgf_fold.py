"""The LGF table and its spectrum (Section 2.2, eq. [lgf_bessel]) where their
kernels change form: Bessel rows on both sides of the switch from Miller's
recurrence to the large-argument series (every N: the nodes reach from t = 0
to 100 N^2), odd table sizes around the blocks of eight entries, many panels
below t = 1 (large s: more nodes than one pass of the table kernel holds), and
the folded cosine transform against the plain sum over the library's own table
from the smallest N to several 32-lane blocks. Tables to 1e-13 of
each entry against the oracle's quadrature, spectra to 1e-12 of the largest
value, the bounds of the other comparisons of both."""
import numpy as np
import pytest

from oracle import lgf as OL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2502_05507_gb300 import Context
    c = Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("N,s", [(2, 0.0), (7, 0.0), (8, 0.3), (9, 0.0), (17, 1e-6), (41, 0.0)])
def test_table_sizes(ctx, N, s):
    got = ctx.lgf_table(N, s)
    ref = OL.lgf_triples(OL.sorted_triples(N), s)
    assert np.all(np.abs(got - ref) <= 1e-13 * np.abs(ref) + 1e-17)


def test_table_with_many_panels_below_one(ctx):
    # s = 1e9: 21 panels below t = 1; G(0) = 1 / (6 + s) (1 + 6 / (6 + s)^2 + ...)
    got = ctx.lgf_table(4, 1e9)
    assert abs(got[0] * (6.0 + 1e9) - 1.0) <= 1e-13


@pytest.mark.parametrize("N,s", [(8, 0.0), (16, 0.01), (32, 0.0), (64, 0.002), (128, 0.0)])
def test_spectrum_is_the_cosine_sum_of_the_table(ctx, N, s):
    t = OL.sorted_triples(N)
    cube = np.zeros((N,) * 3)
    val = ctx.lgf_table(N, s)
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        cube[t[:, p[0]], t[:, p[1]], t[:, p[2]]] = val
    k, n = np.arange(N + 1), np.arange(N)
    C = 2.0 * np.cos(np.pi * ((k[:, None] * n[None, :]) % (2 * N)) / N)
    C[:, 0] = 1.0
    ref = np.einsum("ai,ijk->ajk", C, np.einsum("bj,ijk->ibk", C, cube @ C.T, optimize=True), optimize=True)
    got = ctx.lgf_spectrum(N, s)
    assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref))
