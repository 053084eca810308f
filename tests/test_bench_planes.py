"""The plane count of bench.py's kernel model: the planes that hold sources, which
the applies transform, and not the range that Problem.conv_planes() reports, which
has a plane of margin on each side."""
import numpy as np
import pytest

import bench
import workloads as W
from oracle import grid as OG


@pytest.mark.parametrize("N", [32, 64])
def test_planes_of_the_torus(N):
    P = W.torus_poisson_dir(N, W.torus_batch_dirs(1, seed=3)[0])
    cls = OG.classify(P.phi, P.grid.h, P.grid.origin)
    z = np.flatnonzero(np.any(cls.gm | cls.dnode, axis=(0, 1)))
    reported = (2, int(z[0]) - 1, int(z[-1]) + 2)
    assert bench.transformed_planes(reported) == (2, int(z[-1] - z[0]) + 1)
