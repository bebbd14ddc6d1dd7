"""Timing of the d >= 2 grid stage leaves its kernels as they are."""

import numpy as np
import pytest

import paper_2504_21785_gb300 as fgr

from ._gpu import options, reconstruct, rel_l2

pytestmark = pytest.mark.gpu


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
