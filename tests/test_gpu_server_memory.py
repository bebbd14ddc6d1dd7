"""The server's memory account: buffers that a request can do without are taken only
where the budget has room for them."""

import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
    import math, numpy as np, torch
    import paper_2504_21785_gb300 as fgr
    from workloads import random_packets
    n, eps = 1 << 20, 1 / 1024
    pk = random_packets(5, 1, 16384, q_range=(-3, 3), p_range=(-1, 1), s_range=(-1, 1))
    grid = dict(d=1, n=[n], lo=[-math.pi], hi=[math.pi])
    opt = fgr.make_options(precision=fgr.FGR_FP32)
    u, small = torch.zeros(n, dtype=torch.complex64, device="cuda"), torch.zeros(n, dtype=torch.complex64, device="cuda")
    srv = fgr.fgr_server_create({budget} << 20, 2)
    few = {{k: np.ascontiguousarray(v[..., :4000]) for k, v in pk.items() if k in "qpsa"}}
    ids = [fgr.fgr_register_packets(srv, 1, fgr.make_packets(*[np.ascontiguousarray(x[k]) for k in "qpsa"]))
           for x in (few, pk)]
    fgr.fgr_poll(srv, fgr.fgr_submit(srv, fgr.make_request(0, grid, eps, opt, ids[0], small)), -1)  # loads the kernels
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    res = fgr.fgr_poll(srv, fgr.fgr_submit(srv, fgr.make_request(0, grid, eps, opt, ids[1], u)), -1)
    torch.cuda.synchronize()
    print("TOOK", res.status, before - torch.cuda.mem_get_info()[0])
    fgr.fgr_server_destroy(srv)
"""


@pytest.mark.parametrize("budget,partials", [(24, False), (400, True)])
def test_partial_sums_stay_within_the_budget(budget, partials):
    """16,384 packets onto 2^20 points: at most 24 MB without partial sums, which take 64 MB
    (memory that the library's pool keeps after the call; some of it is there before)."""
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(CODE.format(budget=budget))], cwd=ROOT,
                       env=dict(os.environ, PYTHONPATH=ROOT), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    status, took = [line.split()[1:] for line in r.stdout.splitlines() if line.startswith("TOOK")][0]
    assert status == "0"
    assert (int(took) > 24 << 20) == partials


BATCH = """
    import math, numpy as np, torch
    import paper_2504_21785_gb300 as fgr
    rng = np.random.default_rng(3)
    m = 1 << 20
    pk = [rng.uniform(-0.5, 0.5, (2, m)), rng.uniform(-0.5, 0.5, (2, m)), rng.uniform(-1, 1, m), rng.standard_normal((2, m))]
    opt = fgr.make_options(precision=fgr.FGR_FP32)
    srv = fgr.fgr_server_create(16 << 30, 1)
    ids = [fgr.fgr_register_packets(srv, 2, fgr.make_packets(*pk)),
           fgr.fgr_register_packets(srv, 2, fgr.make_packets(*[np.ascontiguousarray(x[..., :1000]) for x in pk]))]
    grid = dict(d=2, n=[64, 64], lo=[-1, -1], hi=[1, 1])
    slow = dict(d=2, n=[1024, 1024], lo=[-1, -1], hi=[1, 1])
    us = torch.zeros((1024, 1024), dtype=torch.complex64, device="cuda")
    def ask(method, g, eps, i, u):
        return fgr.fgr_submit(srv, fgr.make_request(method, g, eps, opt, ids[i], u))
    # loads the kernels and leaves the direct sum's memory with the pool
    for t in (ask(0, slow, 1 / 64, 0, us), ask(1, grid, 1 / 60, 1, us)):
        assert fgr.fgr_poll(srv, t, -1).status == 0
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    outs = [torch.zeros((64, 64), dtype=torch.complex64, device="cuda") for _ in range(8)]
    tickets = [ask(0, slow, 1 / 64, 0, us)] + [ask(1, grid, 1 / (61 + i), 0, u) for i, u in enumerate(outs)]
    assert all(fgr.fgr_poll(srv, t, -1).status == 0 for t in tickets)
    torch.cuda.synchronize()
    print("TOOK", before - torch.cuda.mem_get_info()[0])
    fgr.fgr_server_destroy(srv)
"""


def test_plans_of_a_batch_hold_no_binning():
    """Eight 2-D requests that wait for a direct sum run as one batch, whose plans take a
    few MB each; binning buffers would add 80 bytes per packet to each."""
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(BATCH)], cwd=ROOT,
                       env=dict(os.environ, PYTHONPATH=ROOT), capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    took = [int(line.split()[1]) for line in r.stdout.splitlines() if line.startswith("TOOK")]
    assert took[0] <= 4 * (80 << 20)
