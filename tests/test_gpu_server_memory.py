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
