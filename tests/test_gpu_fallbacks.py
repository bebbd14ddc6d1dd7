"""Paths that a call takes at the limits of the faster ones: packets outside the FP32
form of the sorted records, memory too short for the binning or the partial sums, and
the row-wise grid passes against the point-wise ones."""

import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

import paper_2504_21785_gb300 as fgr
from workloads import mesh_for

from ._gpu import options, reconstruct, rel_l2, to_device
from .test_gpu_binned import lattice_2d

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _binned(pk, grid, eps, opt):
    """The call's result, and whether it binned its packets."""
    with fgr.Context(grid["d"], grid, eps, opt) as ctx:
        fgr.fgr_set_timing(ctx.handle, 1)
        u = reconstruct("fggc", pk, grid, eps, opt, ctx=ctx)
        return u, fgr.fgr_get_stats(ctx.handle).coeff_ms > 0


def _in_parts(pk, grid, eps, opt):
    """The sum of the results of parts that are too few to be binned."""
    total, step = 0.0, (1 << 17) - 1
    for i in range(0, pk["s"].size, step):
        part = {k: np.ascontiguousarray(pk[k][..., i:i + step]) for k in ("q", "p", "s", "a")}
        u, binned = _binned(part, grid, eps, opt)
        assert not binned
        total = total + u.astype(np.complex128)
    return total


@pytest.mark.parametrize("n_a,n_b,thin", [(26, 30, 0.7), (40, 22, 0.5), (23, 64, 0.15)])
@pytest.mark.parametrize("nq,np_", [(4, 2), (2, 4)])
def test_binned_2d_tiles_of_large_sets(n_a, n_b, thin, nq, np_):
    """Edges of the 24 x 16 tiles, bins of one, two and many items and small bins, on a
    grid that cuts part of the packets off."""
    pk, mesh, eps = lattice_2d(3, n_a, n_b, 0.45, thin)
    grid = dict(d=2, n=[65, 44], lo=[-0.7, -0.5], hi=[1.1, 0.9])
    opt = options("fp32", nq=nq, np_=np_)
    got, binned = _binned(pk, grid, eps, opt)
    assert pk["s"].size >= 1 << 18 and binned
    # both sides round the same contributions and sums to FP32 (2e-7 each)
    assert rel_l2(got, _in_parts(pk, grid, eps, opt)) <= 2e-6


@pytest.mark.parametrize("nq,np_", [(4, 2), (2, 2), (2, 4)])
def test_packet_order_decides_on_2d_binning(nq, np_):
    """The same packets out of order (binned) and in mesh order (too few of them, per
    packet), in a call and through a plan."""
    pk, mesh, eps = lattice_2d(5, 20, 19, 0.4)
    m = pk["s"].size
    assert 1 << 17 <= m < 1 << 18
    cell = [np.floor(x[l] / dx) for l in range(2) for x, dx in ((pk["q"], mesh.dq), (pk["p"], mesh.dp))]
    by_mesh = np.lexsort(cell[::-1])
    grid = dict(d=2, n=[50, 61], lo=[-0.8, -0.7], hi=[0.9, 0.8])
    opt = options("fp32", nq=nq, np_=np_)
    torch = pytest.importorskip("torch")
    out = []
    for idx, want in ((np.arange(m), True), (by_mesh, False)):
        x = {k: np.ascontiguousarray(pk[k][..., idx]) for k in ("q", "p", "s", "a")}
        u, binned = _binned(x, grid, eps, opt)
        assert binned == want
        out.append(u)
        arrays = to_device(x)
        packets = fgr.make_packets(*arrays)
        v = torch.zeros(tuple(grid["n"]), dtype=torch.complex64, device="cuda")
        with fgr.Context(2, grid, eps, opt) as ctx:
            plan = fgr.fgr_fggc_plan_create(ctx.handle, packets, 1)
            fgr.fgr_reconstruct_fggc_planned(ctx.handle, plan, packets, v)
            assert not fgr.fgr_fggc_plan_overflow(plan)
            fgr.fgr_fggc_plan_destroy(plan)
        out.append(v.cpu().numpy())
    # both sides round the same contributions and sums to FP32 (2e-7 each)
    for v in out[1:]:
        assert rel_l2(v, out[0]) <= 2e-6


@pytest.mark.parametrize("shape,binned_whole", [((190, 175, 6, 8), False), ((95, 88, 16, 12), True)])
def test_mesh_order_with_four_neighbours(shape, binned_whole):
    """1.6 million packets in mesh order, Q2P2: binned where bins hold many of them."""
    eps = 1 / 64
    mesh = mesh_for(2, eps)
    rng = np.random.default_rng(12)
    idx = np.indices(shape).reshape(4, -1) + rng.uniform(0.1, 0.9, (4, int(np.prod(shape))))
    idx -= np.array(shape)[:, None] // 2
    m = idx.shape[1]
    pk = {"q": idx[[0, 2]] * mesh.dq, "p": idx[[1, 3]] * mesh.dp, "s": rng.uniform(-1, 1, m),
          "a": rng.standard_normal((2, m))}
    grid = dict(d=2, n=[128, 24], lo=[-6.0, -0.6], hi=[6.0, 0.6])
    opt = options("fp32", nq=2, np_=2)
    got, binned = _binned(pk, grid, eps, opt)
    assert binned == binned_whole
    # both sides round the same contributions and sums to FP32 (2e-7 each)
    assert rel_l2(got, _in_parts(pk, grid, eps, opt)) <= 2e-6


@pytest.mark.parametrize("wide,binned_whole", [(4.0, False), (1.5, True)])
def test_small_bins_out_of_order_stay_per_packet(wide, binned_whole):
    """Packets out of order over an inner plane of half a tile: binned where the
    mean bin is worth it."""
    rng = np.random.default_rng(9)
    m, eps = 1 << 18, 1 / 64
    q = np.stack([rng.uniform(-wide, wide, m), rng.uniform(-0.2, 0.2, m)])
    p = np.stack([rng.uniform(-2 * wide, 2 * wide, m), rng.uniform(-0.2, 0.2, m)])
    pk = {"q": q, "p": p, "s": rng.uniform(-1, 1, m), "a": rng.standard_normal((2, m))}
    grid = dict(d=2, n=[200, 16], lo=[-4.5, -0.3], hi=[4.5, 0.3])
    got, binned = _binned(pk, grid, eps, options("fp32"))
    assert binned == binned_whole
    # both sides round the same contributions and sums to FP32 (2e-7 each)
    assert rel_l2(got, _in_parts(pk, grid, eps, options("fp32"))) <= 2e-6


@pytest.mark.parametrize("shift_a,shift_b,amp,act", [
    (1 << 18, 0, 1.0, 1.0), (-(1 << 18), 0, 1.0, 1.0), (0, 1 << 18, 1.0, 1.0), ((1 << 18) - 10, 3, 1.0, 1.0),
    (60, 40, 1.0, 3e4)])
def test_records_at_the_limits_of_their_fp32_form(shift_a, shift_b, amp, act):
    """Anchors of 2^18 cells and on both sides of it, and actions beyond 2^18 turns, in
    every packet: the binned scatter against parts of the set that are too few to be
    binned."""
    pk, mesh, eps = lattice_2d(6, 26, 21, 0.45)
    for l in range(2):
        pk["q"][l] += shift_a * mesh.dq
        pk["p"][l] += shift_b * mesh.dp
    pk["a"] *= amp
    pk["s"] *= act
    lo = [shift_a * mesh.dq - 0.5, shift_a * mesh.dq - 0.6]
    grid = dict(d=2, n=[40, 36], lo=lo, hi=[lo[0] + 1.1, lo[1] + 1.2])
    got, binned = _binned(pk, grid, eps, options("fp32"))
    assert binned
    # both sides round the same contributions and sums to FP32 (2e-7 each)
    assert rel_l2(got, _in_parts(pk, grid, eps, options("fp32"))) <= 2e-6


@pytest.mark.parametrize("prec,tol", [("fp32", 2e-6), ("fp64", 1e-12)])
@pytest.mark.parametrize("n", [(1, 70), (65, 8), (128, 63), (33, 64), (20, 65, 9), (66, 1, 130)])
@pytest.mark.parametrize("spread", [0.05, 0.9])
def test_row_wise_passes_against_point_wise_ones(n, spread, prec, tol):
    """The edges of the row-wise passes' tiles and ranges, with the other pass kernels
    (pass tile 128) on the same packets."""
    d, eps = len(n), 1 / 64
    rng = np.random.default_rng(8)
    m = 400
    q, p = rng.uniform(-spread, spread, (d, m)), rng.uniform(-0.8, 0.8, (d, m))
    p[0] -= 2 * q[0]
    pk = {"q": q, "p": p, "s": rng.uniform(-1, 1, m), "a": rng.standard_normal((2, m))}
    # (a single point lies at lo)
    lo = [-0.05 if k == 1 else x for k, x in zip(n, (-1.3, -1.1, -0.9))]
    grid = dict(d=d, n=list(n), lo=lo, hi=[1.1, 1.2, 1.3][:d])
    opt = options(prec)
    out, launches = [], []
    for tile in (0, 128):
        with fgr.Context(d, grid, eps, opt) as ctx:
            fgr.fgr_set_tuning(ctx.handle, 8, 16, tile)
            fgr.fgr_set_timing(ctx.handle, 1)
            out.append(reconstruct("fggc", pk, grid, eps, opt, ctx=ctx))
            launches.append(fgr.fgr_get_stats(ctx.handle).launches)
    assert launches[0] != launches[1]
    # FP32: phases and Gaussians per dimension, below 2e-6; FP64: 1e-15 per term
    assert rel_l2(out[0], out[1]) <= tol


# The scratch allocation that a call can do without is the last of its own (8th of a 2-D
# FGGC call, 5th of a 1-D direct sum): it fails once, the next call has it.
@pytest.mark.parametrize("method,d,fail_at", [("fggc", 2, 8), ("direct", 1, 5)])
def test_short_memory_takes_the_path_without_it(method, d, fail_at):
    code = """
        import sys
        sys.path.insert(0, ".")
        import numpy as np
        import paper_2504_21785_gb300 as fgr
        from tests._gpu import options, reconstruct, rel_l2
        rng = np.random.default_rng(2)
        d, m, eps = {d}, 1 << 18, 1 / 64
        pk = {{"q": rng.uniform(-0.4, 0.4, (d, m)), "p": rng.uniform(-0.5, 0.5, (d, m)), "s": rng.uniform(-1, 1, m),
              "a": rng.standard_normal((2, m))}}
        grid = dict(d=d, n=[200, 30][:d], lo=[-0.6] * d, hi=[0.7] * d)
        ctx = fgr.Context(d, grid, eps, options("fp32"))
        fgr.fgr_set_timing(ctx.handle, 1)
        out = []
        for _ in range(2):
            out.append(reconstruct("{method}", pk, grid, eps, options("fp32"), ctx=ctx))
            s = fgr.fgr_get_stats(ctx.handle)
            print("CALL", s.launches, int(s.coeff_ms > 0))
        print("ERR", rel_l2(out[0], out[1]))
    """
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code.format(d=d, method=method))], cwd=ROOT,
                       env=dict(os.environ, FGR_INJECT_ALLOC_FAILURE=str(fail_at), PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    lines = [line.split() for line in r.stdout.splitlines()]
    short, whole = [x for x in lines if x[0] == "CALL"]
    assert short[1] != whole[1]
    if method == "fggc":
        assert (short[2], whole[2]) == ("0", "1")
    # the same FP32 terms in another order of summation
    assert float([x for x in lines if x[0] == "ERR"][0][1]) <= 2e-6
