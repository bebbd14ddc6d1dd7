"""The 1-D FP32 direct sum at the edges of its threads' runs, tiles and slices."""

import numpy as np
import pytest

from oracle import fga
from workloads.wkb import mesh_for

from ._gpu import options, reconstruct, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 1023, 1025, 2051, 5000])
@pytest.mark.parametrize("window_r", [0.0, 2.0, 9.0])
@pytest.mark.parametrize("m", [1, 129, 3000, 4095, 4096])
def test_direct_1d_runs_and_windows(n, window_r, m):
    """Windows that start and end inside a thread's eight points, reach past the grid
    or cover it, zero amplitudes, on both sides of the rules 4 h <= sqrt(eps) and m >= 4096."""
    eps = 1 / 256
    mesh = mesh_for(1, eps)
    rng = np.random.default_rng(n + m)
    a = rng.standard_normal((2, m)) * (rng.random(m) < 0.9)
    pk = {"q": rng.uniform(-1.2, 1.2, (1, m)), "p": rng.uniform(-1, 1, (1, m)), "s": rng.uniform(-1, 1, m), "a": a}
    grid = dict(d=1, n=[n], lo=[-1.0], hi=[1.0])
    got = reconstruct("direct", pk, grid, eps, options("fp32", window_r=window_r))
    ref = fga.direct_sum(pk, grid, eps, mesh.dq, mesh.dp, R=window_r or 6.0)
    # FP32 terms (phase, ex2 and up to four powers: below 2e-6 each), compensated sums
    assert rel_l2(got, ref) <= 4e-6


@pytest.mark.parametrize("window_r", [2.6, 3.4])
def test_direct_1d_few_pairs_per_point(window_r):
    """Both sides of the rule on packet-point pairs: m R sqrt(eps) = 42 and 54 per point
    on a grid of length 2, against the rule's 48."""
    eps, m, n = 1 / 65536, 4096, 5000
    mesh = mesh_for(1, eps)
    rng = np.random.default_rng(n)
    pk = {"q": rng.uniform(-1.0, 1.0, (1, m)), "p": rng.uniform(-1, 1, (1, m)), "s": rng.uniform(-1, 1, m),
          "a": rng.standard_normal((2, m))}
    grid = dict(d=1, n=[n], lo=[-1.0], hi=[1.0])
    got = reconstruct("direct", pk, grid, eps, options("fp32", window_r=window_r))
    ref = fga.direct_sum(pk, grid, eps, mesh.dq, mesh.dp, R=window_r)
    # FP32 terms (phase, ex2 and up to four powers: below 2e-6 each), compensated sums
    assert rel_l2(got, ref) <= 4e-6
