"""The d >= 2 grid stage at the limits of its launches."""

import numpy as np
import pytest

import paper_2504_21785_gb300 as fgr
from oracle import fggc, lsa
from workloads.wkb import mesh_for

from ._gpu import options, reconstruct, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-10)])
def test_outer_plane_of_more_than_a_million_nodes(prec, tol):
    """Packets at the ends of a wide momentum and position range in dimension 0, few
    nodes in dimension 1: more nodes in the outer plane than 65535 groups of 16."""
    eps = 1 / 4096
    mesh = mesh_for(2, eps)
    rng = np.random.default_rng(3)
    m = 40
    q0, p0 = rng.uniform(-3.1, 3.1, m), rng.uniform(-5, 5, m)
    q0[:2], p0[:2] = (-3.1, 3.1), (-5, 5)
    pk = {"q": np.stack([q0, rng.uniform(0.1, 0.9, m) * mesh.dq]), "p": np.stack([p0, rng.uniform(0.1, 0.9, m) * mesh.dp]),
          "s": rng.uniform(-1, 1, m), "a": rng.standard_normal((2, m))}
    nodes = (np.ptp(q0) / mesh.dq) * (np.ptp(p0) / mesh.dp)
    assert nodes > 65535 * 16
    grid = dict(d=2, n=[1021, 5], lo=[-3.2, -0.03], hi=[3.2, 0.04])
    R = 6.0 if prec == "fp32" else 8.0
    got = reconstruct("fggc", pk, grid, eps, options(prec))
    ref = fggc.reconstruct(pk, grid, eps, mesh.dq, mesh.dp, lsa.Strategy(nq=4, np_=2), R=R)
    assert rel_l2(got, ref) <= tol


def test_too_many_points_per_dimension_is_a_capacity_error():
    """More tiles of 64 points than a launch takes: the refusal of the other pass
    kernels, not a launch error, and the context works afterwards."""
    eps = 1 / 64
    pk = {"q": np.zeros((2, 1)), "p": np.zeros((2, 1)), "s": np.zeros(1), "a": np.ones((2, 1))}
    with pytest.raises(fgr.FgrError) as e:
        reconstruct("fggc", pk, dict(d=2, n=[65535 * 64 + 1, 2], lo=[-1, -1], hi=[1, 1]), eps, options("fp32"))
    assert e.value.status == fgr.fgr.FGR_E_CAPACITY
    got = reconstruct("fggc", pk, dict(d=2, n=[40, 30], lo=[-1, -1], hi=[1, 1]), eps, options("fp32"))
    assert np.linalg.norm(got) > 0


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-10)])
@pytest.mark.parametrize("b_nodes", [2, 7, 8, 9, 16, 17, 40])
def test_rows_of_few_and_many_cells(b_nodes, prec, tol):
    """The scan of the node array in groups of 8, 16 and 32 lanes."""
    eps = 1 / 256
    mesh = mesh_for(2, eps)
    rng = np.random.default_rng(b_nodes)
    m = 200
    span = max(0.4, b_nodes - 2.4) * mesh.dp  # (anchors and the neighbour above them)
    q = np.stack([rng.uniform(-0.3, 0.3, m), rng.uniform(-0.2, 0.2, m)])
    p = np.stack([rng.uniform(-0.5, 0.5, m), 0.3 * mesh.dp + rng.uniform(0, span, m)])
    pk = {"q": q, "p": p, "s": rng.uniform(-1, 1, m), "a": rng.standard_normal((2, m))}
    grid = dict(d=2, n=[37, 66], lo=[-0.5, -0.6], hi=[0.6, 0.5])
    R = 6.0 if prec == "fp32" else 8.0
    got = reconstruct("fggc", pk, grid, eps, options(prec))
    ref = fggc.reconstruct(pk, grid, eps, mesh.dq, mesh.dp, lsa.Strategy(nq=4, np_=2), R=R)
    assert rel_l2(got, ref) <= tol


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-10)])
def test_few_rows_of_a_wide_plane(prec, tol):
    """Many nodes in dimension 1 and few in dimension 0: the scan's and the passes' parts
    of a row."""
    eps = 1 / 1024
    mesh = mesh_for(2, eps)
    rng = np.random.default_rng(4)
    m = 60
    q1, p1 = rng.uniform(-3, 3, m), rng.uniform(-4, 4, m)
    q1[:2], p1[:2] = (-3, 3), (-4, 4)
    pk = {"q": np.stack([rng.uniform(0.1, 0.9, m) * mesh.dq, q1]), "p": np.stack([rng.uniform(0.1, 0.9, m) * mesh.dp, p1]),
          "s": rng.uniform(-1, 1, m), "a": rng.standard_normal((2, m))}
    grid = dict(d=2, n=[5, 700], lo=[-0.03, -3.2], hi=[0.04, 3.2])
    R = 6.0 if prec == "fp32" else 8.0
    got = reconstruct("fggc", pk, grid, eps, options(prec))
    ref = fggc.reconstruct(pk, grid, eps, mesh.dq, mesh.dp, lsa.Strategy(nq=4, np_=2), R=R)
    assert rel_l2(got, ref) <= tol
