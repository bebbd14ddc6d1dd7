// Host precomputation of the pseudo-inverse of the eps-free Gram matrix
// (Algorithm 2, Step 0; Remark 2).
//
// The Gram matrix of eq. 3.22 (paper convention, ones on the diagonal)
//   A~_jk = exp(-cq^2/4 (dq_j-dq_k)^2 - cp^2/4 (dp_j-dp_k)^2
//               + i cq cp/2 (dq_k-dq_j)(dp_j+dp_k))
// is Hermitian positive semi-definite, so its SVD is its eigen-decomposition.
// It is computed here by the cyclic complex Jacobi method in long double and
// rounded to double once; singular values below rcond * lambda_max are dropped.
// The device applies the pseudo-inverse through its factors (not the formed
// matrix A~^+), in a basis in which it falls into two real halves.
#include <cmath>
#include <complex>
#include <vector>

#include "internal.h"

namespace fgr {

namespace {
using cld = std::complex<long double>;

void jacobi_hermitian(int n, std::vector<cld> &A, std::vector<cld> &V) {
    V.assign(n * n, cld(0));
    for (int i = 0; i < n; ++i) V[i * n + i] = 1;
    for (int sweep = 0; sweep < 100; ++sweep) {
        long double off = 0, diag = 0;
        for (int i = 0; i < n; ++i)
            for (int j = 0; j < n; ++j) {
                if (i == j)
                    diag += std::norm(A[i * n + j]);
                else
                    off += std::norm(A[i * n + j]);
            }
        if (off <= 1e-40L * diag) break;
        for (int p = 0; p < n - 1; ++p)
            for (int q = p + 1; q < n; ++q) {
                cld apq = A[p * n + q];
                long double mag = std::abs(apq);
                if (mag == 0) continue;
                long double app = A[p * n + p].real(), aqq = A[q * n + q].real();
                // rotation J = [[c, s e], [-s conj(e), c]] on columns p, q with e = apq/|apq|
                cld e = apq / mag;
                long double tau = (aqq - app) / (2 * mag);
                long double t = (tau >= 0 ? 1 : -1) / (std::fabs(tau) + std::sqrt(1 + tau * tau));
                long double c = 1 / std::sqrt(1 + t * t), s = t * c;
                // A <- J^H A J
                for (int k = 0; k < n; ++k) {  // columns
                    cld akp = A[k * n + p], akq = A[k * n + q];
                    A[k * n + p] = c * akp - s * std::conj(e) * akq;
                    A[k * n + q] = s * e * akp + c * akq;
                }
                for (int k = 0; k < n; ++k) {  // rows
                    cld apk = A[p * n + k], aqk = A[q * n + k];
                    A[p * n + k] = c * apk - s * e * aqk;
                    A[q * n + k] = s * std::conj(e) * apk + c * aqk;
                }
                for (int k = 0; k < n; ++k) {
                    cld vkp = V[k * n + p], vkq = V[k * n + q];
                    V[k * n + p] = c * vkp - s * std::conj(e) * vkq;
                    V[k * n + q] = s * e * vkp + c * vkq;
                }
            }
    }
}
}  // namespace

bool build_lsa(double cq, double cp, int nq, int np, double rcond, Lsa *out) {
    static const int s2[2] = {0, 1}, s4[4] = {-1, 0, 1, 2};
    if ((nq != 2 && nq != 4) || (np != 2 && np != 4) || !(cq > 0) || !(cp > 0)) return false;
    const int *sq = nq == 2 ? s2 : s4, *sp = np == 2 ? s2 : s4;
    Lsa L;
    L.nq = nq;
    L.np = np;
    L.n1 = nq * np;
    L.cq = cq;
    L.cp = cp;
    const int n = L.n1;
    for (int iq = 0; iq < nq; ++iq)
        for (int ip = 0; ip < np; ++ip) {
            L.dq[iq * np + ip] = sq[iq];
            L.dp[iq * np + ip] = sp[ip];
        }
    std::vector<cld> A(n * n), V;
    const long double lcq = cq, lcp = cp;
    for (int j = 0; j < n; ++j)
        for (int k = 0; k < n; ++k) {
            long double ddq = L.dq[j] - L.dq[k], ddp = L.dp[j] - L.dp[k];
            long double re = -lcq * lcq / 4 * ddq * ddq - lcp * lcp / 4 * ddp * ddp;
            long double im = lcq * lcp / 2 * (L.dq[k] - L.dq[j]) * (L.dp[j] + L.dp[k]);
            A[j * n + k] = std::exp(re) * cld(std::cos(im), std::sin(im));
        }
    jacobi_hermitian(n, A, V);
    // sort eigenpairs by eigenvalue, descending
    std::vector<int> idx(n);
    for (int i = 0; i < n; ++i) idx[i] = i;
    for (int i = 0; i < n; ++i)
        for (int j = i + 1; j < n; ++j)
            if (A[idx[j] * n + idx[j]].real() > A[idx[i] * n + idx[i]].real()) std::swap(idx[i], idx[j]);
    const long double lmax = A[idx[0] * n + idx[0]].real();
    L.rank = 0;
    for (int i = 0; i < n; ++i) {
        long double lam = A[idx[i] * n + idx[i]].real();
        L.lam[i] = (double)lam;
        if (lam > (long double)rcond * lmax) ++L.rank;
    }
    // Symmetric form of the problem.  With the cell
    // centre as origin and the Weyl-ordered packets D(Q, P) g = e^{i P (x - Q/2)}
    // g(x - Q) as basis, two symmetries of phase space map the neighbour set to
    // itself: parity (x -> -x) and complex conjugation (P -> -P).  In that gauge,
    // with a further e^{-i cq cp u v / 2},
    //   e_k(X, Y) = c~_k(s, t) e^{i (Phi_k - Phi(s, t))} e^{-i cq cp u_k v_k / 2},
    //   Phi(s, t) = -cq cp / 2 (s t + (s - t) / 2),  X = 2 s - 1,  Y = 2 t - 1,
    // the coefficients of the four mirror images of a neighbour (u, v) are
    //   e_(u,v) = f(X, Y),          e_(-u,-v) = f(-X, -Y),
    //   e_(u,-v) = conj f(X, -Y),   e_(-u,v) = conj f(-X, Y),
    // so the problem splits by parity into two halves, each real in a basis of
    // conjugation-invariant vectors (FP64 kernels: the sectors below), and one
    // function per orbit serves four neighbours, through its parts even and odd in
    // X and Y (FP32 kernels): f is interpolated at kCheb x kCheb Chebyshev nodes,
    // the terms up to the total degree are kept, and each parity part is
    // rewritten in powers of X^2 and Y^2 (in FP32 these lose less to rounding
    // than the Chebyshev recurrences: 2.1e-8 against 3.6e-8 rms for Q4P2).
    // Same problem and cut-off as the FP64 path.
    const long double PI = 3.141592653589793238462643383279502884L;
    int orbit_of[kMaxN1 / 4], norb = 0;
    for (int iq = 0; iq < nq / 2; ++iq)
        for (int ip = 0; ip < np / 2; ++ip) {
            const int mq = nq - 1 - iq, mp = np - 1 - ip;
            L.order[4 * norb + 0] = iq * np + ip;
            L.order[4 * norb + 1] = iq * np + mp;
            L.order[4 * norb + 2] = mq * np + ip;
            L.order[4 * norb + 3] = mq * np + mp;
            if (sq[iq] == -1) L.u3 |= 1 << norb;
            if (sp[ip] == -1) L.v3 |= 1 << norb;
            orbit_of[norb++] = iq * np + ip;
        }
    // the Gram matrix in that gauge (without its last factor), its parity sectors in the basis (components over
    // an orbit's four neighbours) even (1,1,1,1)/2, i(1,-1,-1,1)/2, odd
    // (1,1,-1,-1)/2, i(1,-1,1,-1)/2, and their eigen factors
    {
        auto uk = [&](int k) { return L.dq[L.order[k]] - 0.5L; };
        auto vk = [&](int k) { return L.dp[L.order[k]] - 0.5L; };
        auto expi = [](long double x) { return cld(std::cos(x), std::sin(x)); };
        static const int sign[2][2][4] = {{{1, 1, 1, 1}, {1, -1, -1, 1}}, {{1, 1, -1, -1}, {1, -1, 1, -1}}};
        const int h = n / 2;
        for (int s = 0; s < 2; ++s) {
            std::vector<cld> M(h * h), Q;
            for (int a = 0; a < h; ++a)
                for (int b = 0; b < h; ++b) {
                    cld acc = 0;
                    for (int x = 0; x < 4; ++x)
                        for (int y = 0; y < 4; ++y) {
                            const int j = 4 * (a / 2) + x, k = 4 * (b / 2) + y;
                            const long double du = uk(j) - uk(k), dv = vk(j) - vk(k);
                            cld m = std::exp(-lcq * lcq / 4 * du * du - lcp * lcp / 4 * dv * dv) *
                                    expi(lcq * lcp / 2 * (vk(k) * uk(j) - vk(j) * uk(k)));
                            const cld ea = (a % 2 ? cld(0, 1) : cld(1)) * (long double)sign[s][a % 2][x] / 2.0L;
                            const cld eb = (b % 2 ? cld(0, 1) : cld(1)) * (long double)sign[s][b % 2][y] / 2.0L;
                            acc += std::conj(ea) * m * eb;
                        }
                    M[a * h + b] = acc.real();
                }
            jacobi_hermitian(h, M, Q);
            for (int i = 0; i < h; ++i) {
                const long double lam = M[i * h + i].real();
                L.sec_inv[s][i] = lam > (long double)rcond * lmax ? (double)(0.25L / lam) : 0.0;
                for (int a = 0; a < h; ++a) L.sec[s][a * kMaxHalf + i] = (double)Q[a * h + i].real();
                if (s == 0) {  // (the sums over an orbit's ones: 4 in the first of its two components)
                    long double one = 0;
                    for (int a = 0; a < h; a += 2) one += 4 * Q[a * h + i].real();
                    L.sec_one[i] = (double)one;
                }
            }
        }
        for (int o = 0; o < norb; ++o) {
            const cld k = expi(lcq * lcp / 2 * uk(4 * o) * vk(4 * o));
            L.kap_r[o] = (double)k.real();
            L.kap_i[o] = (double)k.imag();
        }
    }
    const int total = n <= 8 ? surrogate_total<8>() : surrogate_total<16>();
    std::vector<cld> val((size_t)norb * kCheb * kCheb);  // f at the nodes
    long double node[kCheb];
    for (int a = 0; a < kCheb; ++a) node[a] = std::cos(PI * (a + 0.5L) / kCheb);
    for (int ia = 0; ia < kCheb; ++ia)
        for (int ib = 0; ib < kCheb; ++ib) {
            const long double s = 0.5L + 0.5L * node[ia], t = 0.5L + 0.5L * node[ib];
            cld f[kMaxN1], y[kMaxN1];
            for (int j = 0; j < n; ++j) {
                long double re = -lcq * lcq / 4 * (L.dq[j] - s) * (L.dq[j] - s) -
                                 lcp * lcp / 4 * (L.dp[j] - t) * (L.dp[j] - t);
                long double im = lcq * lcp / 2 * (s - L.dq[j]) * (L.dp[j] + t);
                f[j] = std::exp(re) * cld(std::cos(im), std::sin(im));
            }
            for (int i = 0; i < n; ++i) {  // y = diag(inv_lam) V^H f
                cld acc = 0;
                for (int j = 0; j < n; ++j) acc += std::conj(V[j * n + idx[i]]) * f[j];
                long double lam = A[idx[i] * n + idx[i]].real();
                y[i] = lam > (long double)rcond * lmax ? acc / lam : cld(0);
            }
            auto phi = [&](long double a, long double b) { return -lcq * lcp / 2 * (a * b + (a - b) / 2); };
            for (int o = 0; o < norb; ++o) {
                const int k = orbit_of[o];
                cld acc = 0;
                for (int i = 0; i < n; ++i) acc += V[k * n + idx[i]] * y[i];
                const long double u = L.dq[k] - 0.5L, v = L.dp[k] - 0.5L;
                const long double g = phi(L.dq[k], L.dp[k]) - phi(s, t) - lcq * lcp / 2 * u * v;
                val[((size_t)o * kCheb + ia) * kCheb + ib] = std::conj(acc) * cld(std::cos(g), std::sin(g));
            }
        }
    // powers of X in T_i(X)
    long double T[kCheb][kCheb] = {};
    T[0][0] = T[1][1] = 1;
    for (int i = 2; i < kCheb; ++i)
        for (int e = 0; e < kCheb; ++e) T[i][e] = (e > 0 ? 2 * T[i - 1][e - 1] : 0) - T[i - 2][e];
    for (int o = 0; o < norb; ++o) {
        cld mono[kCheb][kCheb] = {};
        for (int i = 0; i < kCheb; ++i)
            for (int j = 0; j < kCheb && i + j <= total; ++j) {
                cld c = 0;  // Chebyshev coefficient of T_i(X) T_j(Y)
                for (int ia = 0; ia < kCheb; ++ia)
                    for (int ib = 0; ib < kCheb; ++ib)
                        c += std::cos(i * PI * (ia + 0.5L) / kCheb) * std::cos(j * PI * (ib + 0.5L) / kCheb) *
                             val[((size_t)o * kCheb + ia) * kCheb + ib];
                c *= 4.0L / (kCheb * kCheb) * (i == 0 ? 0.5L : 1.0L) * (j == 0 ? 0.5L : 1.0L);
                for (int e = i; e >= 0; e -= 2)
                    for (int g = j; g >= 0; g -= 2) mono[e][g] += c * T[i][e] * T[j][g];
            }
        for (int e = 0; e < kCheb; ++e)
            for (int g = 0; g < kCheb; ++g) {
                const int part = (e & 1) + 2 * (g & 1);
                float *p = L.poly + o * kOrbitTable + (part * kPow + e / 2) * kPow + g / 2;
                p[0] = (float)mono[e][g].real();
                p[4 * kPow * kPow] = (float)mono[e][g].imag();
            }
    }
    *out = L;
    return true;
}

}  // namespace fgr
