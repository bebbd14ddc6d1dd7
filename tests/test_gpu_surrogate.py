"""The FP32 coefficient surrogate (one polynomial per orbit of mirrored
neighbours) against the FP64 least-squares path of the same library."""

import numpy as np
import pytest

import paper_2504_21785_gb300 as fgr
from workloads.wkb import mesh_for

from ._gpu import options, reconstruct, rel_l2

pytestmark = pytest.mark.gpu

# FP32 rounding of one call: the coefficients (2^-24 times about ten operations),
# two phases reduced to FP32 turns (2^-25 turns = 1.9e-7 rad each) and the grid
# pass's phase and Gaussian (2^-22): below 2e-6 for terms that do not cancel.
TOL = 2e-6


@pytest.mark.parametrize("nq,np_", [(2, 2), (4, 2), (2, 4), (4, 4)])
@pytest.mark.parametrize("d", [1, 2, 3])
def test_surrogate_in_every_part_of_a_cell(d, nq, np_):
    """One packet at a time would do; a handful far apart, at the corners, edges
    and inside of their cells and with anchors of either sign, covers every
    mirror image of every orbit."""
    eps = 1 / 64
    mesh = mesh_for(d, eps)
    frac = np.array([0.0, 1e-7, 0.25, 0.5, 0.75, 1 - 1e-7])
    rng = np.random.default_rng(5 + d)
    m = 36
    q, p = np.empty((d, m)), np.empty((d, m))
    for l in range(d):
        q[l] = (rng.integers(-20, 20, m) + frac[rng.permutation(m) % 6]) * mesh.dq
        p[l] = (rng.integers(-30, 30, m) + frac[rng.permutation(m) % 6]) * mesh.dp
    pk = {"q": q, "p": p, "s": rng.uniform(-1, 1, m), "a": rng.standard_normal((2, m))}
    grid = dict(d=d, n=[97, 61, 33][:d], lo=[-2.0] * d, hi=[2.0] * d)
    ref = reconstruct("fggc", pk, grid, eps, options("fp64", nq, np_, window_r=6.0))
    got = reconstruct("fggc", pk, grid, eps, options("fp32", nq, np_, window_r=6.0))
    assert rel_l2(got, ref) <= TOL


@pytest.mark.parametrize("nq,np_", [(2, 2), (4, 2), (2, 4), (4, 4)])
@pytest.mark.parametrize("d,m", [(1, 40), (1, 9000), (2, 300)])
def test_fp64_factors_against_the_oracle(d, m, nq, np_):
    """The symmetric factors of the FP64 path for every strategy, few packets (small
    CTAs) and many, on ragged grids of the row-wise passes: at the conditioning floor
    of the least-squares problem (its smallest kept singular value)."""
    from oracle import fggc, lsa
    eps = 1 / 64
    mesh = mesh_for(d, eps)
    rng = np.random.default_rng(40 + m)
    pk = {"q": rng.uniform(-0.6, 0.6, (d, m)), "p": rng.uniform(-0.8, 0.8, (d, m)), "s": rng.uniform(-1, 1, m),
          "a": rng.standard_normal((2, m))}
    grid = dict(d=d, n=[83, 41][:d], lo=[-1.1, -0.9][:d], hi=[1.0, 1.2][:d])
    strat = lsa.Strategy(nq=nq, np_=np_)
    sv = strat.pinv.singular_values
    floor = 4 * np.finfo(float).eps / np.sqrt(sv[sv > 1e-14 * sv[0]][-1])
    got = reconstruct("fggc", pk, grid, eps, options("fp64", nq, np_))
    ref = fggc.reconstruct(pk, grid, eps, mesh.dq, mesh.dp, strat, R=8)
    assert rel_l2(got, ref) <= max(1e-12, 2 * floor)  # both sides are at the floor
