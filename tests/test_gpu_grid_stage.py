"""Timing and tuning of the d >= 2 grid stage leave its kernels as they are."""

import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

import paper_2504_21785_gb300 as fgr

from ._gpu import options, reconstruct, rel_l2

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _packets(d, m=500):
    rng = np.random.default_rng(d)
    return {"q": rng.uniform(-0.5, 0.5, (d, m)), "p": rng.uniform(-0.6, 0.6, (d, m)), "s": rng.uniform(-1, 1, m),
            "a": rng.standard_normal((2, m))}


def _call(ctx, pk, grid, eps, opt, level):
    fgr.fgr_set_timing(ctx.handle, level)
    u = reconstruct("fggc", pk, grid, eps, opt, ctx=ctx)
    return u, fgr.fgr_get_stats(ctx.handle)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("d", [2, 3])
def test_counting_terms_times_the_same_kernels(d, prec):
    eps, pk, opt = 1 / 64, _packets(d), options(prec)
    grid = dict(d=d, n=[45, 70, 33][:d], lo=[-1.0] * d, hi=[1.2] * d)
    with fgr.Context(d, grid, eps, opt) as ctx:
        u1, s1 = _call(ctx, pk, grid, eps, opt, 1)
        u2, s2 = _call(ctx, pk, grid, eps, opt, 2)
        fgr.fgr_set_tuning(ctx.handle, 8, 16, 128)  # the point-wise passes
        _, s3 = _call(ctx, pk, grid, eps, opt, 2)
    assert s1.launches == s2.launches != s3.launches
    # (one order of atomic additions against another)
    assert rel_l2(u2, u1) <= (1e-6 if prec == "fp32" else 1e-12)
    # the same lines and ranges, but for values that underflow
    assert s2.pass_terms > 0 and abs(s2.pass_terms - s3.pass_terms) <= 0.01 * s3.pass_terms


def test_tuned_tile_does_not_replace_the_row_wise_passes(tmp_path):
    path = tmp_path / "tune.txt"
    path.write_text("2 %d 9 12 8 16 128\n" % fgr.FGR_FP32)
    code = """
        import sys
        sys.path.insert(0, ".")
        import paper_2504_21785_gb300 as fgr
        from tests.test_gpu_grid_stage import _call, _packets, options
        eps, pk, opt = 1 / 64, _packets(2), options("fp32")
        grid = dict(d=2, n=[45, 70], lo=[-1.0] * 2, hi=[1.2] * 2)
        ctx = fgr.Context(2, grid, eps, opt)
        print("TUNING", *fgr.fgr_get_tuning(ctx.handle))
        print("TUNED", _call(ctx, pk, grid, eps, opt, 1)[1].launches)
        for tile in (0, 32, 128):
            fgr.fgr_set_tuning(ctx.handle, 8, 16, tile)
            print("SET", _call(ctx, pk, grid, eps, opt, 1)[1].launches)
    """
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, FGR_TUNE_FILE=str(path), PYTHONPATH=ROOT), timeout=300)
    assert r.returncode == 0, r.stderr
    out = [line.split() for line in r.stdout.splitlines() if line.split()[0] in ("TUNING", "TUNED", "SET")]
    assert out[0][1:] == ["8", "16", "128"]
    tuned, default, tile32, tile128 = (int(x[1]) for x in out[1:])
    assert tuned == default == tile32 != tile128


def test_autotune_keeps_what_the_row_wise_passes_do_not_use():
    import torch
    from ._gpu import to_device
    eps, pk, opt = 1 / 64, _packets(2), options("fp32")
    grid = dict(d=2, n=[45, 70], lo=[-1.0] * 2, hi=[1.2] * 2)
    with fgr.Context(2, grid, eps, opt) as ctx:
        fgr.fgr_set_tuning(ctx.handle, 8, 23, 0)
        arrs = to_device(pk)
        u = torch.zeros((45, 70), dtype=torch.complex64, device="cuda")
        fgr.fgr_autotune(ctx.handle, fgr.make_packets(*arrs), u, 2)
        assert fgr.fgr_get_tuning(ctx.handle) == (8, 23, 0)
        assert rel_l2(u.cpu().numpy(), reconstruct("fggc", pk, grid, eps, opt)) <= 1e-6
