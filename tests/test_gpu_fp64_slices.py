"""FP64 1-D FGGC on either side of the grid pass's rules on tiles and slices."""

import numpy as np
import pytest

from oracle import fggc, lsa
from workloads.wkb import mesh_for

from ._gpu import options, reconstruct, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [97, 2200, 2600, 5000, 7700, 9001])
@pytest.mark.parametrize("spread", [0.2, 3.0])
def test_tiles_and_slices(n, spread):
    """Grids of 1 to 71 tiles of 128 points, with nodes on a part of them and on all:
    narrow tiles in slices of 8, wide ones in slices of 16 and 32 b values."""
    eps = 1 / 64
    mesh = mesh_for(1, eps)
    rng = np.random.default_rng(n)
    m = 500
    pk = {"q": rng.uniform(-spread, spread, (1, m)), "p": rng.uniform(-1.5, 1.5, (1, m)), "s": rng.uniform(-1, 1, m),
          "a": rng.standard_normal((2, m))}
    grid = dict(d=1, n=[n], lo=[-3.1], hi=[3.0])
    pts = rng.integers(0, n, (1, 300))
    got = reconstruct("fggc", pk, grid, eps, options("fp64"))
    ref = fggc.reconstruct(pk, grid, eps, mesh.dq, mesh.dp, lsa.Strategy(nq=4, np_=2), R=8, points=pts)
    # the oracle's rounding over the square root of its smallest singular value: 8.6e-12
    assert rel_l2(got[tuple(pts)], ref) <= 2e-11
