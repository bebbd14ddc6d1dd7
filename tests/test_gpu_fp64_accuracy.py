"""FP64 FGGC against the same least-squares problem in extended precision: the
rounding of the right-hand side, which the small eigenvalues of the Gram matrix
divide, stays far below FP64's own."""

import numpy as np
import pytest

from oracle import fga

from ._gpu import options, reconstruct, rel_l2

pytestmark = pytest.mark.gpu

LD, CLD = np.longdouble, np.clongdouble


def _expi(x):
    return np.cos(x) + 1j * np.sin(x)


def _eigen(A):
    """Eigenvalues and eigenvectors of a Hermitian matrix by Jacobi rotations."""
    A, n = A.copy(), len(A)
    V = np.eye(n).astype(CLD)
    for _ in range(60):
        off = sum(abs(A[i, j]) ** 2 for i in range(n) for j in range(n) if i != j)
        if off <= 1e-38 * sum(abs(A[i, i]) ** 2 for i in range(n)):
            break
        for p in range(n - 1):
            for q in range(p + 1, n):
                m = abs(A[p, q])
                if m < 1e-300:
                    continue
                e, tau = A[p, q] / m, (A[q, q].real - A[p, p].real) / (2 * m)
                t = (1 if tau >= 0 else -1) / (abs(tau) + np.hypot(LD(1), tau))
                c = 1 / np.sqrt(1 + t * t)
                J = np.eye(n).astype(CLD)
                J[p, p] = J[q, q] = c
                J[p, q], J[q, p] = t * c * e, -t * c * np.conj(e)
                A, V = J.conj().T @ A @ J, V @ J
    return np.array([A[i, i].real for i in range(n)]), V


def _reference(pk, x, eps, dq, dp, cq, cp, nq, np_):
    sets = {2: (0, 1), 4: (-1, 0, 1, 2)}
    kq = np.array([a for a in sets[nq] for _ in sets[np_]], LD)
    kp = np.array([b for _ in sets[nq] for b in sets[np_]], LD)
    cq, cp, dq, dp, eps = (LD(v) for v in (cq, cp, dq, dp, eps))
    D, E = kq[:, None] - kq[None], kp[:, None] - kp[None]
    gram = np.exp(-cq * cq / 4 * D * D - cp * cp / 4 * E * E) * _expi(cq * cp / 2 * -D * (kp[:, None] + kp[None]))
    lam, V = _eigen(gram.astype(CLD))
    u = np.zeros(x.size, CLD)
    for j in range(pk["s"].size):
        r, rp = LD(pk["q"][0, j]) / dq, LD(pk["p"][0, j]) / dp
        a0, b0 = np.floor(r), np.floor(rp)
        s, t = r - a0, rp - b0
        f = np.exp(-cq * cq / 4 * (kq - s) ** 2 - cp * cp / 4 * (kp - t) ** 2) * _expi(cq * cp / 2 * (s - kq) * (kp + t))
        c = np.conj(V @ ((V.conj().T @ f) / lam)) * _expi(-cq * cp * (s - kq) * b0)
        w = (LD(pk["a"][0, j]) + 1j * LD(pk["a"][1, j])) * _expi(LD(pk["s"][j]) / eps)
        for k in range(kq.size):
            y = x - (a0 + kq[k]) * dq
            u += w * c[k] * np.exp(-y * y / (2 * eps)) * _expi((b0 + kp[k]) * dp * y / eps)
    return fga.prefactor(1, float(eps), float(dq), float(dp)) * u, float(lam.min())


# f - 1 and its few roundings: below 2^-55 on the default mesh (f within 1/2 of one, the
# series of small arguments), 2^-53 on wide ones (the library's functions)
@pytest.mark.parametrize("nq,np_,cq,cp,rounding", [
    (2, 2, 0.5, np.pi / 8, 2.0 ** -55), (4, 2, 0.5, np.pi / 8, 2.0 ** -55), (2, 4, 0.5, np.pi / 8, 2.0 ** -55),
    (4, 2, 0.51, 0.6, 2.0 ** -53), (4, 2, 1.0, 1.0, 2.0 ** -53), (2, 2, 1.5, 1.2, 2.0 ** -53)])
def test_least_squares_rounding(nq, np_, cq, cp, rounding):
    if np.finfo(LD).eps > 1e-18:
        pytest.skip("no extended precision")
    eps = 1 / 64
    dq, dp = cq * eps ** 0.5, cp * eps ** 0.5
    rng = np.random.default_rng(17)
    m = 240
    pk = {"q": rng.uniform(-4, 4, (1, m)) * dq, "p": rng.uniform(-4, 4, (1, m)) * dp,
          "s": rng.uniform(-0.02, 0.02, m), "a": rng.standard_normal((2, m))}
    n = 48
    grid = dict(d=1, n=[n], lo=[-0.5], hi=[0.5])
    got = reconstruct("fggc", pk, grid, eps, options("fp64", nq, np_, window_r=20.0, cq=cq, cp=cp))
    x = LD(-0.5) + np.arange(n).astype(LD) / n
    ref, lam = _reference(pk, x, eps, dq, dp, cq, cp, nq, np_)
    err = rel_l2(got, ref.astype(np.complex128))
    print("Q%dP%d cq %.2f cp %.2f: %.2e" % (nq, np_, cq, cp, err))
    # over the square root of the smallest eigenvalue; phases, Gaussians and sums of the
    # grid pass: 2e-15
    assert err <= rounding / lam ** 0.5 + 2e-15
