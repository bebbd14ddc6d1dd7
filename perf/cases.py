"""The calls that a user of the library makes, as measurable cases.

A case names an operation, its sizes and its options as plain values.
`prepare` builds what a program has in hand before the call (packets on the
device, context, plan, output buffer), `run` makes the call through the C ABI
binding, and `exact` gives the same result in 64 bits from plain torch.

Inputs.  The packets are the WKB decompositions of the paper's Sec. 4 on its
phase-space meshes (dq = sqrt(eps)/2, dp = pi sqrt(eps)/8): per dimension a wave
exp(-12.5 (x - x0)^2 + i S0(x)/eps) is decomposed on nq x np nodes and carried
along its Hamiltonian flow, so q, p, s and a spread and bend as propagated
packets do.  The seed moves the wave's centre and momentum, its phase and the
propagation time.  All potentials of the library are separable, so a d-dim set
is the product of d per-dimension lists; that is also what makes a 64-bit
result cheap.
"""

import math

import numpy as np
import torch

import paper_2504_21785_gb300 as fgr

CQ, CP = 0.5, math.pi / 8
TAU = 2 * math.pi


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest reconstruction: 4096 packets in double precision on 1024
        # points, where launches and the one host wait count
        dict(name="fggc_1d_f64_small", op="fggc", d=1, inv_eps=64, nq=64, np=64, n0=1024, prec="f64",
             sq=4, sp=2, t=0.5),
        # the 1-D workload of the benchmark
        dict(name="fggc_1d", op="fggc", d=1, inv_eps=1024, nq=512, np=512, n0=32768, prec="f32", sq=4, sp=2, t=1.0),
        # the 2-D workload: 4.2M packets onto 1024^2 points
        dict(name="fggc_2d", op="fggc", d=2, inv_eps=256, nq=64, np=32, n0=1024, n1=1024, prec="f32",
             sq=4, sp=2, t=0.5),
        # double precision and the small neighbour set on an odd grid, as in the
        # error studies of Sec. 4
        dict(name="fggc_2d_f64_odd", op="fggc", d=2, inv_eps=64, nq=40, np=21, n0=301, n1=257, prec="f64",
             sq=2, sp=2, t=0.5),
        # the headline: 2^24 packets onto 256^3 points
        dict(name="fggc_3d", op="fggc", d=3, inv_eps=64, nq=32, np=16, cap=1 << 24, n0=256, n1=256, n2=256,
             prec="f32", sq=4, sp=2, t=0.5),
        # a small 3-D preview on a ragged grid: few packets per phase-space cell
        dict(name="fggc_3d_small", op="fggc", d=3, inv_eps=64, nq=20, np=10, cap=300001, n0=96, n1=81, n2=100,
             prec="f32", sq=4, sp=2, t=0.5),
        # windowed direct sums, the method's reference result: 1-D and 2-D
        # workloads, and a ragged 3-D grid
        dict(name="direct_1d", op="direct", d=1, inv_eps=1024, nq=512, np=512, n0=32768, prec="f32", t=1.0),
        dict(name="direct_2d", op="direct", d=2, inv_eps=256, nq=64, np=32, n0=1024, n1=1024, prec="f32", t=0.5),
        dict(name="direct_3d", op="direct", d=3, inv_eps=64, nq=24, np=12, cap=1 << 21, n0=200, n1=180, n2=171,
             prec="f32", t=0.5),
        # packet propagation over a tenth of a time unit: 1000 RK4 steps
        dict(name="propagate_1d", op="propagate", d=1, inv_eps=1024, nq=512, np=512, t=0.1, steps=1000),
        # multi-step evolution on a tensor-product mesh: decomposition, learned
        # flow and FGGC per step, at the 2-D workload's sizes
        dict(name="multistep_2d", op="multistep", d=2, inv_eps=256, nq=64, np=32, n0=1024, n1=1024, prec="f32",
             sq=4, sp=2, t=0.25, steps=2),
        # a serving step: 32 planned 1-D reconstructions of mixed size in one call
        dict(name="batch_fggc_1d", op="batch", d=1, requests=32, m_min=4096, m_max=65536, n_min=1024, n_max=32768,
             prec="f32", sq=4, sp=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above."""
    op, d = rng.choice([("fggc", 1), ("fggc", 1), ("fggc", 2), ("fggc", 2), ("fggc", 3), ("fggc", 3),
                        ("direct", 1), ("direct", 2), ("direct", 3), ("propagate", 1), ("multistep", 1),
                        ("multistep", 2), ("batch", 1)])
    if op == "batch":
        return dict(op=op, d=1, requests=rng.randint(2, 48), m_min=_log_int(rng, 1024, 4096),
                    m_max=_log_int(rng, 8192, 65536), n_min=_log_int(rng, 512, 2048),
                    n_max=_log_int(rng, 4096, 32768), prec="f32", sq=4, sp=rng.choice([2, 2, 4]))
    c = dict(op=op, d=d, inv_eps=_log_int(rng, 64, (1024, 400, 100)[d - 1]))
    if op == "propagate":
        return c | dict(nq=_log_int(rng, 64, 512), np=_log_int(rng, 64, 512), t=round(rng.uniform(0.02, 0.1), 3),
                        steps=_log_int(rng, 100, 1000))
    top = 512 if d == 1 else (64 if d == 2 else (32 if op == "fggc" else 24))
    c["nq"] = _log_int(rng, (64, 24, 14)[d - 1], top)
    c["np"] = _log_int(rng, (32, 12, 7)[d - 1], top if d == 1 else top // 2)
    if d == 3:
        most = min((1 << 24) if op == "fggc" else (1 << 20), (c["nq"] * c["np"]) ** 3)
        c["cap"] = _log_int(rng, min(1 << 16, most), most)
    for l in range(d):
        c["n%d" % l] = _log_int(rng, (1000, 128, 64)[d - 1], (32768, 1024, 256 if op == "fggc" else 180)[d - 1])
    c["prec"] = rng.choice(["f32", "f32", "f64"]) if op == "fggc" and d < 3 else "f32"
    if op == "multistep":
        c["steps"] = rng.randint(1, 4)
    c["t"] = round(rng.uniform(0.1, 1.0 if d == 1 else 0.5), 3)
    if op != "direct":
        c["sq"], c["sp"] = rng.choice([(4, 2), (4, 2), (2, 2)])
        if c["prec"] == "f64":  # the double-precision path solves per packet: fewer of them
            c["nq"], c["np"] = min(c["nq"], 256 if d == 1 else 40), min(c["np"], 128 if d == 1 else 21)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _flow(kind, q, p, t, steps):
    """Eq. 2.3-2.6 for one dimension by RK4, from unit amplitude: Q, P, S and the
    complex amplitude factor.  kind: V = 1 - cos x or V = x^2/2."""
    if kind == "harmonic":
        c, s = math.cos(t), math.sin(t)
        Q, P = q * c + p * s, p * c - q * s
        S = 0.5 * (P * Q - p * q)
        return Q, P, S, torch.polar(torch.ones_like(q), torch.full_like(q, -t / 2))

    def rhs(y):
        Q, P, _, F, G, H, K = y  # F = dQ/dq, G = dQ/dp, H = dP/dq, K = dP/dp
        v, dv, ddv = 1 - torch.cos(Q), torch.sin(Q), torch.cos(Q)
        return P, -dv, 0.5 * P * P - v, H, K, -ddv * F, -ddv * G

    one, zero = torch.ones_like(q), torch.zeros_like(q)
    y = (q, p, zero, one, zero, zero, one)
    h = t / steps
    last, turns = torch.zeros_like(q), torch.zeros_like(q)
    for _ in range(steps):
        k1 = rhs(y)
        k2 = rhs(tuple(a + 0.5 * h * b for a, b in zip(y, k1)))
        k3 = rhs(tuple(a + 0.5 * h * b for a, b in zip(y, k2)))
        k4 = rhs(tuple(a + h * b for a, b in zip(y, k3)))
        y = tuple(a + h / 6 * (b1 + 2 * b2 + 2 * b3 + b4) for a, b1, b2, b3, b4 in zip(y, k1, k2, k3, k4))
        arg = torch.atan2(y[5] - y[4], y[3] + y[6])  # Z = (F + K) + i (H - G), Z(0) = 2
        turns += torch.round((last - arg) / TAU)
        last = arg
    Q, P, S, F, G, H, K = y
    mag, arg = torch.hypot(F + K, H - G) / 2, last + TAU * turns
    return Q, P, S, torch.polar(torch.sqrt(mag), arg / 2)


def _wave(case, l, rng):
    """(centre, momentum, phase) of the wave along dimension l."""
    return rng.uniform(-0.05, 0.05), rng.uniform(-0.1, 0.1), rng.uniform(0, TAU)


def _s0(d, l, kick, y):
    """S0 and its derivative along dimension l: a focusing front, or a plane wave (d = 3)."""
    if d == 3:
        return (1 + kick) * y, torch.full_like(y, 1 + kick)
    if l == 0:
        z = 5 * y
        return -(z.abs() + torch.log1p(torch.exp(-2 * z.abs()))) / 5 + kick * y, kick - torch.tanh(z)
    return kick * y, torch.full_like(y, kick)


def _mesh_dim(d, l, eps, nq, np_, wave, dev):
    """One dimension's mesh and amplitudes at t = 0: q, p, A (nq * np entries, a-major)."""
    x0, kick, phase = wave
    dq, dp = CQ * math.sqrt(eps), CP * math.sqrt(eps)
    q = (torch.arange(nq, dtype=torch.float64, device=dev) - nq // 2) * dq
    beta = torch.round(_s0(d, l, kick, q)[1] / dp)[:, None] + (
        torch.arange(np_, dtype=torch.float64, device=dev)[None, :] - np_ // 2)
    L = max(256, 1 << (4 * np_ - 1).bit_length())
    h = TAU * eps / (dp * L)
    k = torch.arange(-L // 2, L // 2, dtype=torch.float64, device=dev)
    y = q[:, None] + k[None, :] * h
    f = torch.polar(torch.exp(-12.5 * (y - x0) ** 2 - ((k * h) ** 2 / (2 * eps))[None, :]),
                    _s0(d, l, kick, y)[0] / eps + phase)
    spec = torch.fft.fft(torch.roll(f, L // 2, 1), dim=1) * h
    amp = math.sqrt(2.0) * torch.gather(spec, 1, torch.remainder(beta, L).long())
    return q.repeat_interleave(np_), (beta * dp).reshape(-1), amp.reshape(-1)


class _Set:
    """A propagated packet set: per-dimension lists and the kept products."""

    def __init__(self, case, seed, flow_only=False):
        rng = np.random.default_rng([seed, 17])
        dev = _device()
        self.d, self.eps = case["d"], 1.0 / case["inv_eps"]
        d = self.d
        t = case["t"] * rng.uniform(0.95, 1.05)
        kind = "harmonic" if d == 3 else "cosine"
        self.q0, self.p0, self.a0, self.dims = [], [], [], []
        for l in range(d):
            q, p, a = _mesh_dim(d, l, self.eps, case["nq"], case["np"], _wave(case, l, rng), dev)
            Q, P, S, f = _flow(kind, q, p, t, 64)
            self.q0.append(q)
            self.p0.append(p)
            self.a0.append(a)
            self.dims.append((Q, P, S, f if flow_only else a * f))
        self.shape = (case["nq"],) * d + (case["np"],) * d
        self.kept = None
        if "cap" in case:  # the largest amplitudes, in mesh order
            mag = self._product([x[3].abs().float() for x in self.dims], torch.mul)
            self.kept = torch.topk(mag, case["cap"], sorted=False).indices.sort().values

    def _spread(self, l, v):
        """v of dimension l's list over the packets' (a_1..a_d, b_1..b_d) index."""
        s = [1] * (2 * self.d)
        s[l], s[self.d + l] = self.shape[l], self.shape[self.d + l]
        return v.reshape(self.shape[l], self.shape[self.d + l]).reshape(s)

    def _product(self, vs, f):
        x = self._spread(0, vs[0])
        for l in range(1, self.d):
            x = f(x, self._spread(l, vs[l]))
        return x.expand(self.shape).reshape(-1)

    def _keep(self, x):
        return (x if self.kept is None else x[self.kept]).contiguous()

    def index(self, l):
        """Entry of dimension l's list of every kept packet."""
        n = self.shape[l] * self.shape[self.d + l]
        i = torch.arange(n, device=self.dims[0][0].device)
        return self._keep(self._spread(l, i).expand(self.shape).reshape(-1))

    def tensor_index(self):
        """Row-major index of every packet in the product of the d lists."""
        L = self.shape[0] * self.shape[self.d]
        sel = self.index(0)
        for l in range(1, self.d):
            sel = sel * L + self.index(l)
        return sel.contiguous()

    def arrays(self):
        """q (d, M), p (d, M), s (M), a (2, M) in double precision."""
        m = self.kept.numel() if self.kept is not None else int(np.prod(self.shape))
        dev = self.dims[0][0].device
        q = torch.empty((self.d, m), dtype=torch.float64, device=dev)
        p, a = torch.empty_like(q), torch.empty((2, m), dtype=torch.float64, device=dev)
        for l in range(self.d):
            q[l] = self._keep(self._spread(l, self.dims[l][0]).expand(self.shape).reshape(-1))
            p[l] = self._keep(self._spread(l, self.dims[l][1]).expand(self.shape).reshape(-1))
        s = self._keep(self._product([x[2] for x in self.dims], torch.add))
        amp = self._keep(self._product([x[3] for x in self.dims], torch.mul))
        a[0], a[1] = amp.real, amp.imag
        return q, p, s, a


def _grid(case):
    d = case["d"]
    return dict(d=d, n=[case["n%d" % l] for l in range(d)], lo=[-math.pi] * d, hi=[math.pi] * d)


def _options(case):
    return fgr.make_options(precision=fgr.FGR_FP64 if case["prec"] == "f64" else fgr.FGR_FP32,
                            nq=case.get("sq", 4), np_=case.get("sp", 2))


def _complex(case):
    return torch.complex128 if case["prec"] == "f64" else torch.complex64


def _field(case, seed):
    """The wave that a multi-step evolution starts from, on the grid (64-bit complex values
    of the case's precision)."""
    rng = np.random.default_rng([seed, 17])
    rng.uniform(0.95, 1.05)
    dev, d, eps, u = _device(), case["d"], 1.0 / case["inv_eps"], None
    for l in range(d):
        x0, kick, phase = _wave(case, l, rng)
        x = _points(case, l, dev)
        f = torch.polar(torch.exp(-12.5 * (x - x0) ** 2), _s0(d, l, kick, x)[0] / eps + phase)
        u = f if u is None else u[..., None] * f
    return u.to(_complex(case)).contiguous()


def _batch_cases(case, seed):
    """The requests of a batch: each its own set, eps and grid."""
    rng = np.random.default_rng([seed, 23, case["requests"]])
    size = np.random.default_rng([7, case["requests"], case["m_max"], case["n_max"]])  # sizes by the case alone
    out = []
    for _ in range(case["requests"]):
        m = math.exp(size.uniform(math.log(case["m_min"]), math.log(case["m_max"])))
        np_ = int(size.integers(32, 129))
        n = int(round(math.exp(size.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        inv = int(round(math.exp(size.uniform(math.log(64), math.log(1024)))))
        out.append((dict(op="fggc", d=1, inv_eps=inv, nq=max(16, int(m / np_)), np=np_, n0=n, prec=case["prec"],
                         sq=case["sq"], sp=case["sp"], t=0.5), int(rng.integers(1 << 30))))
    return out


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

_streams = {}


def _stream():
    """The stream that the calls are made on."""
    if "s" not in _streams:
        _streams["s"] = torch.cuda.Stream()
    return _streams["s"]


class _State:
    """Everything a program keeps between calls; plans are freed with it."""

    def __init__(self, **kw):
        self.plans = []
        self.__dict__.update(kw)

    def __del__(self):
        for p in self.plans:
            fgr.fgr_fggc_plan_destroy(p)


def prepare(case, seed):
    op = case["op"]
    dev = _device()
    if op == "batch":
        s = _State(op=op, stream=_stream(), ctx=[], packets=[], u=[])
        for sub, sub_seed in _batch_cases(case, seed):
            pk = fgr.make_packets(*_Set(sub, sub_seed).arrays())
            torch.cuda.synchronize()  # the plan reads the packets on another stream
            s.ctx.append(fgr.Context(1, _grid(sub), 1.0 / sub["inv_eps"], _options(sub)))
            s.packets.append(pk)
            s.u.append(torch.empty(sub["n0"], dtype=_complex(sub), device=dev))
            s.plans.append(fgr.fgr_fggc_plan_create(s.ctx[-1].handle, pk, 2, s.stream))
        s.handles = [c.handle for c in s.ctx]
        return s
    if op == "propagate":
        x = _Set(dict(case, t=1.0), seed, flow_only=True)
        q, p, a = x.q0[0][None].contiguous(), x.p0[0][None].contiguous(), torch.stack([x.a0[0].real, x.a0[0].imag])
        start = (q, p, torch.zeros_like(q[0]), a.contiguous())
        now = tuple(torch.empty_like(v) for v in start)
        grid = dict(d=1, n=[1024], lo=[-math.pi], hi=[math.pi])
        return _State(op=op, stream=_stream(), ctx=fgr.Context(1, grid, x.eps), start=start, now=now,
                      packets=fgr.make_packets(*now), pot=fgr.make_potential("cossum", c0=1.0, amp=-1.0),
                      t=case["t"], dt=case["t"] / case["steps"])
    grid, eps = _grid(case), 1.0 / case["inv_eps"]
    x = _Set(case, seed, flow_only=op == "multistep")
    s = _State(op=op, stream=_stream(), ctx=fgr.Context(case["d"], grid, eps, _options(case)),
               packets=fgr.make_packets(*x.arrays()), u=torch.empty(grid["n"], dtype=_complex(case), device=dev))
    if op == "multistep":
        s.u0, s.steps = _field(case, seed), case["steps"]
        s.axes = fgr.make_axes(list(zip(x.q0, x.p0)))
        s.sel = x.tensor_index()
    return s


def run(s):
    if s.op == "fggc":
        fgr.fgr_reconstruct_fggc(s.ctx.handle, s.packets, s.u, s.stream)
    elif s.op == "direct":
        fgr.fgr_reconstruct_direct(s.ctx.handle, s.packets, s.u, s.stream)
    elif s.op == "multistep":
        fgr.fgr_fggc_multistep_tensor(s.ctx.handle, s.axes, s.sel, s.packets, s.u0, s.u, s.steps, s.stream)
    elif s.op == "batch":
        fgr.fgr_reconstruct_fggc_batch(s.handles, s.plans, s.packets, s.u, s.stream)
    else:  # propagation works in place: the packets at t = 0 are kept
        with torch.cuda.stream(s.stream):
            for to, of in zip(s.now, s.start):
                to.copy_(of)
        fgr.fgr_propagate(s.ctx.handle, s.packets, s.pot, s.t, s.dt, s.stream)
        return dict(zip("qpsa", s.now))
    return s.u


# ---------------------------------------------------------------------------
# work: what a pass cannot do without
# ---------------------------------------------------------------------------

def _fggc_work(case):
    """Packets read, grid written; contributions (one complex multiply-add each)
    and, per dimension, the contraction of the nodes a window reaches (one
    complex multiply-add per node and point)."""
    d, n1 = case["d"], case["sq"] * case["sp"]
    m = case.get("cap", (case["nq"] * case["np"]) ** d)
    n = [case["n%d" % l] for l in range(d)]
    out = math.prod(n) * (16 if case["prec"] == "f64" else 8)
    R = 8 if case["prec"] == "f64" else 6
    terms, nodes = 0.0, case["nq"] * case["np"]
    for l in reversed(range(d)):
        terms += nodes ** l * math.prod(n[l:]) * (2 * R / CQ) * case["np"]
    return dict(bytes=8.0 * m * (2 * d + 3) + out, flops=8.0 * m * n1 ** d + 8.0 * terms)


def work(case):
    op, d = case["op"], case["d"]
    if op == "fggc":
        return _fggc_work(case)
    if op == "batch":
        w = [_fggc_work(c) for c, _ in _batch_cases(case, 0)]
        return dict(bytes=sum(x["bytes"] for x in w), flops=sum(x["flops"] for x in w))
    m = case.get("cap", (case["nq"] * case["np"]) ** d)
    if op == "propagate":  # 4 stages of about 40 operations a step
        return dict(bytes=2 * 40.0 * m, flops=160.0 * m * case["steps"])
    n = [case["n%d" % l] for l in range(d)]
    window = 1.0
    for l in range(d):  # points of a packet's window of 6 sqrt(eps) on either side
        window *= min(n[l], 12 / math.sqrt(case["inv_eps"]) * n[l] / TAU + 1)
    if op == "direct":
        return dict(bytes=8.0 * m * (2 * d + 3) + 8.0 * math.prod(n), flops=8.0 * m * window)
    w = _fggc_work(case)
    entries = case["nq"] * case["np"]
    dec = sum(entries ** (d - l) * math.prod(n[:l]) * window ** (1 / d) for l in range(d)) * 8.0
    field = math.prod(n) * (16 if case["prec"] == "f64" else 8)
    return dict(bytes=case["steps"] * (w["bytes"] + field), flops=case["steps"] * (w["flops"] + dec))


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

def _points(case, l, dev):
    n = case["n%d" % l]
    return -math.pi + torch.arange(n, dtype=torch.float64, device=dev) * (TAU / n)


def _window(case, l, q, eps):
    """First and last grid index of the windows |x - q| <= R sqrt(eps)."""
    n = case["n%d" % l]
    h, r = TAU / n, (8 if case["prec"] == "f64" else 6) * math.sqrt(eps)
    return (torch.ceil((q - r + math.pi) / h).clamp(min=0).long(),
            torch.floor((q + r + math.pi) / h).clamp(max=n - 1).long())


def _functions(case, l, q, p, eps):
    """G(x; q, p) of every entry on the grid of dimension l, zero outside its window: (entries, n)."""
    x = _points(case, l, q.device)
    lo, hi = _window(case, l, q, eps)
    m = torch.arange(x.numel(), device=q.device)
    dx = x[None, :] - q[:, None]
    f = torch.polar(torch.exp(-dx * dx / (2 * eps)), p[:, None] * dx / eps)
    return torch.where((m[None, :] >= lo[:, None]) & (m[None, :] <= hi[:, None]), f, torch.zeros_like(f))


def _shifts(case):
    of = {2: (0, 1), 4: (-1, 0, 1, 2)}
    return [(a, b) for a in of[case["sq"]] for b in of[case["sp"]]]


def _coefficients(case, q, p, eps):
    """Least-squares coefficients of a packet on its grid neighbours, one dimension
    (eq. 3.22-3.23 and the shift back of eq. 3.13): a, b (entries) and c (entries, n1)."""
    sh = np.array(_shifts(case), dtype=np.float64)
    dj, ej, dk, ek = sh[:, 0][:, None], sh[:, 1][:, None], sh[:, 0][None], sh[:, 1][None]
    gram = np.exp(-CQ * CQ / 4 * (dj - dk) ** 2 - CP * CP / 4 * (ej - ek) ** 2
                  + 0.5j * CQ * CP * (dk - dj) * (ej + ek))
    U, S, Vh = np.linalg.svd(gram)
    keep = S > 1e-14 * S[0]
    U, S, V = (torch.from_numpy(np.ascontiguousarray(v)).to(q.device)
               for v in (U[:, keep], S[keep], Vh[keep].conj().T))
    r, rp = q / (CQ * math.sqrt(eps)), p / (CP * math.sqrt(eps))
    a, b = torch.floor(r), torch.floor(rp)
    s, t = (r - a)[:, None], (rp - b)[:, None]
    dk, ek = (torch.from_numpy(np.ascontiguousarray(sh[:, i])).to(q.device)[None] for i in (0, 1))
    f = torch.polar(torch.exp(-CQ * CQ / 4 * (dk - s) ** 2 - CP * CP / 4 * (ek - t) ** 2),
                    0.5 * CQ * CP * (s - dk) * (ek + t))
    c = ((f @ U.conj()) / S) @ V.T
    return a, b, c.conj() * torch.polar(torch.ones_like(s), -CQ * CP * (s - dk) * b[:, None])


def _fitted(case, l, q, p, eps):
    """The on-grid fit of every entry's function on the grid of dimension l: (entries, n)."""
    a, b, c = _coefficients(case, q, p, eps)
    out = 0
    for k, (da, db) in enumerate(_shifts(case)):
        out = out + c[:, k, None] * _functions(case, l, (a + da) * (CQ * math.sqrt(eps)),
                                               (b + db) * (CP * math.sqrt(eps)), eps)
    return out


def _prefactor(case, eps):
    return (CQ * CP * eps / (TAU * eps) ** 1.5) ** case["d"]


def _direct_1d(case, q, p, w, eps):
    """Sum of w G(x; q, p) over the packets, window by window."""
    x = _points(case, 0, q.device)
    u = torch.zeros((2, x.numel()), dtype=torch.float64, device=q.device)
    lo, hi = _window(case, 0, q, eps)
    width = int((hi - lo).max()) + 1
    step = max(1, (1 << 25) // max(width, 1))
    for i in range(0, q.numel(), step):
        j = slice(i, i + step)
        m = lo[j, None] + torch.arange(width, device=q.device)
        ok = m <= hi[j, None]
        m = m.clamp(max=x.numel() - 1)
        dx = x[m] - q[j, None]
        f = torch.polar(torch.exp(-dx * dx / (2 * eps)), p[j, None] * dx / eps) * w[j, None]
        f = torch.where(ok, f, torch.zeros_like(f))
        u[0].index_add_(0, m.reshape(-1), f.real.reshape(-1))
        u[1].index_add_(0, m.reshape(-1), f.imag.reshape(-1))
    return torch.complex(u[0], u[1])


def _fggc_1d(case, q, p, w, eps):
    """The packets' coefficients summed on the nodes, the nodes summed on the grid."""
    a, b, c = _coefficients(case, q, p, eps)
    c = c * w[:, None]
    dq, dp = CQ * math.sqrt(eps), CP * math.sqrt(eps)
    a0, b0 = int(a.min()) - 1, int(b.min()) - 1
    A, B = int(a.max()) + 3 - a0, int(b.max()) + 3 - b0
    W = torch.zeros((2, A * B), dtype=torch.float64, device=q.device)
    for k, (da, db) in enumerate(_shifts(case)):
        i = ((a + da - a0) * B + (b + db - b0)).long()
        W[0].index_add_(0, i, c[:, k].real.contiguous())
        W[1].index_add_(0, i, c[:, k].imag.contiguous())
    na = (torch.arange(A, device=q.device, dtype=torch.float64) + a0) * dq
    nb = (torch.arange(B, device=q.device, dtype=torch.float64) + b0) * dp
    W = torch.complex(W[0], W[1]).reshape(A, B) * torch.polar(
        torch.ones((A, B), dtype=torch.float64, device=q.device), -na[:, None] * nb[None] / eps)
    x = _points(case, 0, q.device)
    E = torch.polar(torch.ones((x.numel(), B), dtype=torch.float64, device=q.device), x[:, None] * nb[None] / eps)
    g = _functions(case, 0, na, torch.zeros_like(na), eps).real
    return ((E @ W.T) * g.T).sum(1)


def _tables(case, x, fit):
    """Per dimension the functions of the list's entries, (entries, n)."""
    return [(_fitted if fit else _functions)(case, l, x.dims[l][0], x.dims[l][1], x.eps) for l in range(x.d)]


def _reconstruction(case, x, fit):
    eps = x.eps
    w = [D[3] * torch.polar(torch.ones_like(D[2]), D[2] / eps) for D in x.dims]
    if x.d == 1:
        return _prefactor(case, eps) * (_fggc_1d if fit else _direct_1d)(case, x.dims[0][0], x.dims[0][1], w[0], eps)
    F = [f * v[:, None] for f, v in zip(_tables(case, x, fit), w)]
    if x.kept is None:
        u = F[0].sum(0)
        for l in range(1, x.d):
            u = u[..., None] * F[l].sum(0)
        return _prefactor(case, eps) * u
    L = F[0].shape[0]  # three dimensions, kept products only
    mask = torch.zeros(L ** 3, dtype=torch.bool, device=w[0].device)
    mask[x.tensor_index()] = True
    mask = mask.reshape(L, L, L)
    U = torch.stack([F[1].T @ (mask[i].to(torch.complex128) @ F[2]) for i in range(L)])
    u = F[0].T @ U.reshape(L, -1)
    return _prefactor(case, eps) * u.reshape([case["n%d" % l] for l in range(3)])


def _multistep(case, seed):
    x = _Set(case, seed, flow_only=True)
    eps, d = x.eps, x.d
    u = _field(case, seed).to(torch.complex128)
    scale = math.prod(math.sqrt(2.0) * TAU / case["n%d" % l] for l in range(d))
    if d == 1:
        q, p, lo_hi = x.q0[0], x.p0[0], _window(case, 0, x.q0[0], eps)
        w = x.dims[0][3] * torch.polar(torch.ones_like(q), x.dims[0][2] / eps)
        X = _points(case, 0, q.device)
        width = int((lo_hi[1] - lo_hi[0]).max()) + 1
        for _ in range(case["steps"]):
            a, step = [], max(1, (1 << 25) // max(width, 1))
            for i in range(0, q.numel(), step):
                j = slice(i, i + step)
                m = lo_hi[0][j, None] + torch.arange(width, device=q.device)
                ok, m = m <= lo_hi[1][j, None], m.clamp(max=X.numel() - 1)
                dx = X[m] - q[j, None]
                f = torch.polar(torch.exp(-dx * dx / (2 * eps)), -p[j, None] * dx / eps) * u[m]
                a.append(torch.where(ok, f, torch.zeros_like(f)).sum(1))
            u = _prefactor(case, eps) * _fggc_1d(case, x.dims[0][0], x.dims[0][1], scale * torch.cat(a) * w, eps)
        return u
    into = [_functions(case, l, x.q0[l], x.p0[l], eps).conj() for l in range(d)]
    back = [f * (D[3] * torch.polar(torch.ones_like(D[2]), D[2] / eps))[:, None]
            for f, D in zip(_tables(case, x, True), x.dims)]
    for _ in range(case["steps"]):
        a = scale * (into[0] @ u @ into[1].T)
        u = _prefactor(case, eps) * (back[0].T @ a @ back[1])
    return u


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        return [_reconstruction(c, _Set(c, s), True) for c, s in _batch_cases(case, seed)]
    if op == "multistep":
        return _multistep(case, seed)
    if op == "propagate":
        x = _Set(dict(case, t=1.0), seed, flow_only=True)
        Q, P, S, f = _flow("cosine", x.q0[0], x.p0[0], case["t"], 500)
        a = x.a0[0] * f
        return dict(q=Q[None], p=P[None], s=S, a=torch.stack([a.real, a.imag]))
    return _reconstruction(case, _Set(case, seed), op == "fggc")
