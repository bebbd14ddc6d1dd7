"""FP32 direct sums where a run of points evaluated by recurrences would start far
from the packet's centre: grids coarser than the Gaussian, and wide windows."""

import numpy as np
import pytest

import paper_2504_21785_gb300 as fgr
from oracle import fga
from workloads.wkb import mesh_for

from ._gpu import options, reconstruct, rel_l2, to_device

pytestmark = pytest.mark.gpu

# FP32 terms: phase, ex2 and the recurrences, below 2e-6 per dimension and factor
# (the tensor-core path's split operands included)
TOL = 1e-5

def _case(d, steps, seed, m=300):
    """Packets on a grid with step steps[l] sqrt(eps) in dimension l."""
    eps = 1 / 256
    sig = eps ** 0.5
    rng = np.random.default_rng(seed)
    n = [(300, 60, 24)[d - 1] if st < 1 else 23 for st in steps]
    lo = [-0.5 * k * st * sig for k, st in zip(n, steps)]
    hi = [0.5 * k * st * sig for k, st in zip(n, steps)]
    q = np.stack([rng.uniform(1.1 * a, 1.1 * b, m) for a, b in zip(lo, hi)])
    # a few on grid points, so that no coarse point is left with tails alone
    for l in range(d):
        q[l, ::3] = lo[l] + rng.integers(0, n[l], q[l, ::3].size) * (hi[l] - lo[l]) / n[l] + 0.1 * sig
    pk = {"q": q, "p": rng.uniform(-1, 1, (d, m)), "s": rng.uniform(-1, 1, m), "a": rng.standard_normal((2, m))}
    return pk, dict(d=d, n=n, lo=lo, hi=hi), eps


@pytest.mark.parametrize("flags", [0, fgr.FGR_FLAG_DIRECT_FMA])
@pytest.mark.parametrize("steps", [(1.1,), (2.3,), (2.4,), (4.6,), (2.6, 0.3), (0.2, 4.6), (7.0, 7.0), (2.3, 2.4), (4.6, 0.3, 2.6), (0.9, 1.1, 0.9)])
@pytest.mark.parametrize("window_r", [6.0, 20.0])
def test_coarse_grids_and_wide_windows(steps, window_r, flags):
    d = len(steps)
    pk, grid, eps = _case(d, steps, 7)
    mesh = mesh_for(d, eps)
    got = reconstruct("direct", pk, grid, eps, options("fp32", window_r=window_r, flags=flags))
    ref = fga.direct_sum(pk, grid, eps, mesh.dq, mesh.dp, R=window_r)
    assert np.all(np.isfinite(got))
    assert rel_l2(got, ref) <= TOL


@pytest.mark.parametrize("window_r", [9.0, 9.5, 13.0, 40.0])
@pytest.mark.parametrize("step", [0.12, 0.13, 0.5])
def test_wide_windows_on_fine_grids(step, window_r):
    """Both sides of the tensor-core rule on windows and steps (h = sqrt(eps) / 8)."""
    pk, grid, eps = _case(2, (step, step), 8)
    mesh = mesh_for(2, eps)
    got = reconstruct("direct", pk, grid, eps, options("fp32", window_r=window_r))
    ref = fga.direct_sum(pk, grid, eps, mesh.dq, mesh.dp, R=window_r)
    assert rel_l2(got, ref) <= TOL


@pytest.mark.parametrize("d", [1, 2])
@pytest.mark.parametrize("steps", [(0.2, 0.1, 0.25), (0.2, 1.5, 4.6, 0.9)])
def test_batched_direct_on_fine_and_coarse_grids(d, steps):
    """A batch of fine grids, and one with grids on either side of the rule."""
    import torch
    reqs = [_case(d, (st,) * d, 20 + i) for i, st in enumerate(steps)]
    ctxs = [fgr.Context(d, g, eps, options("fp32")) for _, g, eps in reqs]
    try:
        arrs = [to_device(pk) for pk, _, _ in reqs]
        pks = [fgr.make_packets(*x) for x in arrs]
        us = [torch.zeros(tuple(g["n"]), dtype=torch.complex64, device="cuda") for _, g, _ in reqs]
        fgr.fgr_reconstruct_direct_batch([c.handle for c in ctxs], pks, us)
        torch.cuda.synchronize()
        for (pk, g, eps), u in zip(reqs, us):
            mesh = mesh_for(d, eps)
            ref = fga.direct_sum(pk, g, eps, mesh.dq, mesh.dp, R=6)
            assert rel_l2(u.cpu().numpy(), ref) <= TOL
    finally:
        for c in ctxs:
            c.close()
