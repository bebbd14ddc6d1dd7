// K3+K4: FGGC coefficients and scatter (Algorithm 2 Step 3, eq. 2.25).
// Included by fggc_coeff1.cu / fggc_coeff2.cu / fggc_coeff3.cu, one per
// dimension, so the heavily unrolled instantiations compile in parallel.
// See fggc.cu for the layout of the node array and the folded node phase.
#pragma once

#include "device_util.cuh"
#include "fggc_params.h"

namespace fgr {
namespace {

// ---------------------------------------------------------------------------
// coefficients + scatter
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cmul(double ar, double ai, double br, double bi, double &cr, double &ci) {
    cr = ar * br - ai * bi;
    ci = ar * bi + ai * br;
}
__device__ __forceinline__ void cmul(float ar, float ai, float br, float bi, float &cr, float &ci) {
    cr = ar * br - ai * bi;
    ci = ar * bi + ai * br;
}

// Parameter views of one request inside a batch: that request's constants
// with the least-squares tables shared by the batch (same strategy).
struct Params64View {
    const Common &c;
    const Factors64 &f;
};
struct Params32View {
    const Common &c;
    const float *poly;
};

// e^x - 1 for -1/4 <= x <= 0 (about an ulp): the Taylor series to x^13, whose next term
// is below 2^-62 of the first.
__device__ __forceinline__ double expm1_near(double x) {
    double p = 1.0 / 6227020800.0;
    p = fma(p, x, 1.0 / 479001600.0);
    p = fma(p, x, 1.0 / 39916800.0);
    p = fma(p, x, 1.0 / 3628800.0);
    p = fma(p, x, 1.0 / 362880.0);
    p = fma(p, x, 1.0 / 40320.0);
    p = fma(p, x, 1.0 / 5040.0);
    p = fma(p, x, 1.0 / 720.0);
    p = fma(p, x, 1.0 / 120.0);
    p = fma(p, x, 1.0 / 24.0);
    p = fma(p, x, 1.0 / 6.0);
    p = fma(p, x, 0.5);
    return fma(p * x, x, x);
}

// Sine and cosine for |x| <= 3/32 (about an ulp): Taylor to x^9 and x^8, whose next
// terms are below 2^-59 and 2^-55.
__device__ __forceinline__ void sincos_near(double x, double &sn, double &cs) {
    const double z = x * x;
    double p = fma(1.0 / 362880.0, z, -1.0 / 5040.0), q = fma(1.0 / 40320.0, z, -1.0 / 720.0);
    p = fma(p, z, 1.0 / 120.0);
    q = fma(q, z, 1.0 / 24.0);
    p = fma(p, z, -1.0 / 6.0);
    q = fma(q, z, -0.5);
    sn = fma(p * z, x, x);
    cs = fma(q, z, 1.0);
}

// e^{x + i y} - 1 from e = e^x - 1 and the sine and cosine of y / 2.
__device__ __forceinline__ void exp_minus_one(double e, double sn_half, double cs_half, double &re, double &im) {
    const double q = 2.0 * sn_half * sn_half;  // 1 - cos y
    re = fma(-(1.0 + e), q, e);
    im = (1.0 + e) * (2.0 * sn_half * cs_half);
}

// FP64: the coefficients of one dimension through the eigen factors (PT: Params64
// or Params64View), in the symmetric form of build_lsa: with (sx, ty) the offset
// from the cell centre, the right-hand side of neighbour (u, v) is
//   e^{-cq^2 (u - sx)^2 / 4} e^{i cq cp u ty / 2} e^{-cp^2 (v - ty)^2 / 4} e^{-i cq cp v sx / 2},
// one exponential per u and per v and a sine and cosine per |u| and per |v| for all
// neighbours; sums and differences of mirror images bring it to the sectors' real
// bases.  All of it is carried as f - 1: the problem's small eigenvalues divide the
// rounding of f by up to their square root (2.6e-5 for Q4P2), f lies near one, and the
// ones' share of every eigenvector is exact (Lsa::sec_one).  Relative to the result,
// random packets: 3.6e-12 for Q4P2 with products of exponentials (3.4e-12 with one
// exponential and phase per neighbour), 3.4e-13 so.  The phases are those of
// dim_setup32: z = e^{i cq cp A / 2}, and T takes the packet's share in turns.  The
// FP64 pipe binds (16 clocks of an SM per warp instruction): against an exponential,
// two sines and cosines and two complex matrix rows per neighbour, 705,600 2-D Q2P2
// packets take 1.73 -> 0.95 ms (1-D, 4096 Q4P2: 66 -> 27 us).
template <int N, class PT>
__device__ __forceinline__ void coeff_dim64(const PT &P, double Q, double Pm, int &a0, int &b0, double &T,
                                            double *cr, double *ci) {
    const Common &c = P.c;
    const double r = __ddiv_rn(Q, c.dqv), rp = __ddiv_rn(Pm, c.dpv);
    const double fa = floor(r), fb = floor(rp);
    const double sx = (r - fa) - 0.5, ty = (rp - fb) - 0.5;
    a0 = (int)fmin(fmax(fa, -1e9), 1e9);
    b0 = (int)fmin(fmax(fb, -1e9), 1e9);
    {
        double t = c.cc * (r * (fb + 0.5));
        t -= rint(t);
        T -= t + 0.5 * c.cc * (sx * ty);
    }
    double zr, zi;
    {
        double t = 0.5 * c.cc * (fa + 0.5);
        t -= rint(t);
        sincospi(2.0 * t, &zi, &zr);
    }
    // Gaussian and phase factors of u, v = -1/2, 1/2 and (where the strategy has
    // them) -3/2, 3/2, less one
    double ur[2][2], ui[2][2], vr2[2][2], vi2[2][2];
    auto factors = [&](auto expm1_of, auto sincos_of) {
#pragma unroll
        for (int t = 0; t < (N >= 8 ? 2 : 1); ++t) {
            const double h = t + 0.5;
            double sn, cs;
            if (t == 0 || c.u3) {
                sincos_of(h * c.cqcp_4 * ty, sn, cs);
                exp_minus_one(expm1_of(-c.cq2_4 * ((h + sx) * (h + sx))), -sn, cs, ur[t][0], ui[t][0]);
                exp_minus_one(expm1_of(-c.cq2_4 * ((h - sx) * (h - sx))), sn, cs, ur[t][1], ui[t][1]);
            }
            if (t == 0 || c.v3) {
                sincos_of(h * c.cqcp_4 * sx, sn, cs);
                exp_minus_one(expm1_of(-c.cp2_4 * ((h + ty) * (h + ty))), sn, cs, vr2[t][0], vi2[t][0]);
                exp_minus_one(expm1_of(-c.cp2_4 * ((h - ty) * (h - ty))), -sn, cs, vr2[t][1], vi2[t][1]);
            }
        }
    };
    if (P.f.near)
        factors([](double x) { return expm1_near(x); }, [](double x, double &s, double &c) { sincos_near(x, s, c); });
    else
        factors([](double x) { return expm1(x); }, [](double x, double &s, double &c) { sincos(x, &s, &c); });
    double gr[2][N / 2], gi[2][N / 2];
#pragma unroll
    for (int o = 0; o < N / 4; ++o) {
        const bool u3 = N >= 8 && ((c.u3 >> o) & 1), v3 = N >= 8 && ((c.v3 >> o) & 1);
        double br[4], bi[4];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int a = g >> 1, b = g & 1;
            const double pr = u3 ? ur[N >= 8 ? 1 : 0][a] : ur[0][a], pi = u3 ? ui[N >= 8 ? 1 : 0][a] : ui[0][a];
            const double qr = v3 ? vr2[N >= 8 ? 1 : 0][b] : vr2[0][b], qi = v3 ? vi2[N >= 8 ? 1 : 0][b] : vi2[0][b];
            // (1 + p) (1 + q) - 1
            br[g] = fma(-pi, qi, fma(pr, qr, pr + qr));
            bi[g] = fma(pr, qi, fma(pi, qr, pi + qi));
        }
        const double pr = br[0] + br[3], pi = bi[0] + bi[3], qr = br[1] + br[2], qi = bi[1] + bi[2];
        gr[0][2 * o] = pr + qr;
        gi[0][2 * o] = pi + qi;
        gr[0][2 * o + 1] = pi - qi;
        gi[0][2 * o + 1] = qr - pr;
        const double mr = br[0] - br[3], mi = bi[0] - bi[3], nr = br[1] - br[2], ni = bi[1] - bi[2];
        gr[1][2 * o] = mr + nr;
        gi[1][2 * o] = mi + ni;
        gr[1][2 * o + 1] = mi - ni;
        gi[1][2 * o + 1] = nr - mr;
    }
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        double wr[N / 2], wi[N / 2];
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            double tr = s == 0 ? P.f.one[i] : 0.0, ti = 0;
#pragma unroll
            for (int a = 0; a < N / 2; ++a) {
                tr = fma(P.f.sec[s][a * kMaxHalf + i], gr[s][a], tr);
                ti = fma(P.f.sec[s][a * kMaxHalf + i], gi[s][a], ti);
            }
            wr[i] = tr * P.f.inv[s][i];
            wi[i] = ti * P.f.inv[s][i];
        }
#pragma unroll
        for (int a = 0; a < N / 2; ++a) {
            double tr = 0, ti = 0;
#pragma unroll
            for (int i = 0; i < N / 2; ++i) {
                tr = fma(P.f.sec[s][a * kMaxHalf + i], wr[i], tr);
                ti = fma(P.f.sec[s][a * kMaxHalf + i], wi[i], ti);
            }
            gr[s][a] = tr;
            gi[s][a] = ti;
        }
    }
#pragma unroll
    for (int o = 0; o < N / 4; ++o) {
        // x1 + i x2 and x1 - i x2 of the even half, y1 + i y2 and y1 - i y2 of the odd
        const double er = gr[0][2 * o] - gi[0][2 * o + 1], ei = gi[0][2 * o] + gr[0][2 * o + 1];
        const double fr = gr[0][2 * o] + gi[0][2 * o + 1], fi = gi[0][2 * o] - gr[0][2 * o + 1];
        const double hr = gr[1][2 * o] - gi[1][2 * o + 1], hi = gi[1][2 * o] + gr[1][2 * o + 1];
        const double lr = gr[1][2 * o] + gi[1][2 * o + 1], li = gi[1][2 * o] - gr[1][2 * o + 1];
        double vr = zr, vi = zi;
        if (N >= 8 && ((c.v3 >> o) & 1)) {
            double r2, i2;
            cmul(zr, zi, zr, zi, r2, i2);
            cmul(r2, i2, zr, zi, vr, vi);
        }
        // e^{-i cq cp v (A + u / 2)} of u < 0 and of u > 0, for v < 0
        double p0r, p0i, p1r, p1i;
        cmul(vr, vi, P.f.kap_r[o], -P.f.kap_i[o], p0r, p0i);
        cmul(vr, vi, P.f.kap_r[o], P.f.kap_i[o], p1r, p1i);
        cmul(er + hr, ei + hi, p0r, p0i, cr[4 * o], ci[4 * o]);
        cmul(fr + lr, fi + li, p0r, -p0i, cr[4 * o + 1], ci[4 * o + 1]);
        cmul(fr - lr, fi - li, p1r, p1i, cr[4 * o + 2], ci[4 * o + 2]);
        cmul(er - hr, ei - hi, p1r, -p1i, cr[4 * o + 3], ci[4 * o + 3]);
    }
}

// FP32: the coefficients by the surrogate of Lsa::poly.  Per dimension, with
// r = Q/dq, the cell centre (A, B) = (a0, b0) + 1/2, sx = r - A, ty = P/dp - B and
// the neighbour's (u, v) = (dq_k, dp_k) - 1/2, the coefficient times the node
// phase is (eq. 3.13 and the gauge of build_lsa)
//   e_k(2 sx, 2 ty) e^{-i cq cp A v} e^{-i cq cp (r B + sx ty / 2)}:
// the last factor does not depend on the neighbour and joins the packet's
// weight (one sine and cosine for the packet), and A v takes two conjugate
// values per orbit (one sine and cosine per dimension).  An orbit of four
// neighbours costs two real polynomials of 72 terms instead of eight.
// Against a pair of 72-term polynomials and a sine and cosine per neighbour
// (1312 multiply-adds of a packet's 1700 instructions per dimension, now about
// 500 in all): 3-D workload (16.8M packets) scatter 9.80 -> 7.45 ms, 1-D (262k)
// 0.049 -> 0.026 ms, 2-D (4.2M) 1.15 -> 1.02 ms, where the reductions bind.

// One dimension of a packet: anchor, surrogate arguments, z = e^{i cq cp A / 2},
// and its share of the packet's phase (rB: sum of r B; xy: sum of sx ty).
__device__ __forceinline__ void dim_setup32(const Common &c, double Q, double Pm, int &a0, int &b0, float &X,
                                            float &Y, float &zr, float &zi, double &rB, float &xy) {
    // the floors of Q/dq and P/dp as the FP64 division decides them (FP32
    // estimate, FP64 only near an integer); the offsets from one FP64 product
    // each (within a few ulps of the quotient, which is all FP32 can resolve)
    a0 = floor_div_int(Q, c.dqv, c.inv_dq);
    b0 = floor_div_int(Pm, c.dpv, c.inv_dp);
    const double A = (double)a0 + 0.5, B = (double)b0 + 0.5;
    const double r = Q * c.inv_dq;
    const float sx = (float)(r - A), ty = (float)fma(Pm, c.inv_dp, -B);
    X = 2.f * sx;
    Y = 2.f * ty;
    rB = fma(r, B, rB);
    xy = fmaf(sx, ty, xy);
    double tz = 0.5 * c.cc * A;
    tz -= rint(tz);
    sincospif(2.f * (float)tz, &zi, &zr);
}

// Weight of a packet: pref A e^{i S/eps} times the neighbour-independent phase.
__device__ __forceinline__ void packet_weight32(const Common &c, double s, double ar, double ai, double rB, float xy,
                                                float &wr, float &wi) {
    double t = fma(-c.cc, rB, s * c.inv_2pi_eps);
    t -= rint(t);
    float sn, cs;
    sincospif(2.f * fmaf(-0.5f * (float)c.cc, xy, (float)t), &sn, &cs);
    cmul((float)(ar * c.pref), (float)(ai * c.pref), cs, sn, wr, wi);
}

// Parity part (PX, PY) of a surrogate polynomial over X^PX Y^PY, in powers of
// xx = X^2 and yy = Y^2 (Horner; the terms of total degree surrogate_total).
// One multiply-add per coefficient, which it reads from the constant bank; the
// packed form (real and imaginary part at once) needs them in registers.
template <int N1, int PX, int PY>
__device__ __forceinline__ float parity_part(const float *C, float xx, float yy) {
    constexpr int T = surrogate_total<N1>();
    float r = 0.f;
#pragma unroll
    for (int i = kPow - 1; i >= 0; --i) {
        const int jtop = (T - 2 * i - PX - PY) / 2 < kPow - 1 ? (T - 2 * i - PX - PY) / 2 : kPow - 1;
        float u = C[i * kPow + jtop];
#pragma unroll
        for (int j = kPow - 1; j >= 0; --j)
            if (j < jtop) u = fmaf(u, yy, C[i * kPow + j]);
        r = i == kPow - 1 ? u : fmaf(r, xx, u);
    }
    return r;
}

// f(X, Y), f(X, -Y), f(-X, Y), f(-X, -Y) of one orbit's polynomial: its four
// coefficients up to the conjugation of the middle two.
template <int N1>
__device__ __forceinline__ void orbit_values(const float *C, float X, float Y, float2 *f) {
    static_assert(surrogate_total<N1>() >= 2 * kPow, "every power of X^2 has a term");
    constexpr int kPart = kPow * kPow;
    const float xx = X * X, yy = Y * Y, xy = X * Y;
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // real, imaginary part
        const float *H = C + h * 4 * kPart;
        const float ee = parity_part<N1, 0, 0>(H, xx, yy), oe = X * parity_part<N1, 1, 0>(H + kPart, xx, yy);
        const float eo = parity_part<N1, 0, 1>(H + 2 * kPart, xx, yy), oo = parity_part<N1, 1, 1>(H + 3 * kPart, xx, yy);
        const float p = fmaf(xy, oo, ee), n = fmaf(-xy, oo, ee), m = fmaf(Y, eo, oe), o = fmaf(-Y, eo, oe);
        const float v[4] = {p + m, n + o, n - o, p - m};
#pragma unroll
        for (int g = 0; g < 4; ++g) (h == 0 ? f[g].x : f[g].y) = v[g];
    }
}

// e^{i cq cp A |v|} of an orbit from z = e^{i cq cp A / 2}.
template <int N1>
__device__ __forceinline__ void orbit_phase(const Common &c, int o, float zr, float zi, float &vr, float &vi) {
    vr = zr;
    vi = zi;
    if (N1 >= 8 && ((c.v3 >> o) & 1)) {
        float r2, i2;
        cmul(zr, zi, zr, zi, r2, i2);
        cmul(r2, i2, zr, zi, vr, vi);
    }
}

// All coefficients of one dimension, times the phases that depend on the
// neighbour and a factor (yr, yi): out(k, re, im).
template <int N1, class PT, class Out>
__device__ __forceinline__ void coeff_dim32(const PT &P, float X, float Y, float zr, float zi, float yr, float yi,
                                            Out out) {
#pragma unroll
    for (int o = 0; o < N1 / 4; ++o) {
        float2 f[4];
        float vr, vi, hr[2], hi[2];
        orbit_values<N1>(P.poly + o * kOrbitTable, X, Y, f);
        orbit_phase<N1>(P.c, o, zr, zi, vr, vi);
        cmul(yr, yi, vr, vi, hr[0], hi[0]);
        cmul(yr, yi, vr, -vi, hr[1], hi[1]);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            float re, im;
            cmul(f[g].x, g == 1 || g == 2 ? -f[g].y : f[g].y, hr[g & 1], hi[g & 1], re, im);
            out(4 * o + g, re, im);
        }
    }
}

// The last dimension's N1 contributions of one row of outer neighbours,
// scaled by (pr, pi): cell idx + (a0 + dq_k - amin) sa + (b0 + dp_k - bmin) sb.
template <int L, int N1, class Real, class C2>
__device__ __forceinline__ void emit_row(C2 *__restrict__ W, const Common &c, int a0, int b0, const Real *cl_r,
                                         const Real *cl_i, int64_t idx, Real pr, Real pi) {
#pragma unroll
    for (int k = 0; k < N1; ++k) {
        const int ia = a0 + c.dq[k] - c.amin[L], ib = b0 + c.dp[k] - c.bmin[L];
        if ((unsigned)ia < (unsigned)c.A[L] && (unsigned)ib < (unsigned)c.B[L]) {
            Real vr, vi;
            cmul(pr, pi, cl_r[k], cl_i[k], vr, vi);
            atomic_add_c(W + idx + ia * c.sa[L] + ib * c.sb[L], vr, vi);
        }
    }
}

// Threads per CTA of the scatter kernel: the coefficients of all dimensions
// but the last wait in shared memory ([dim][neighbour][thread], at most 32 KB).
template <bool FP64, int N1>
__host__ __device__ constexpr int coeff_threads() {
    return (FP64 && N1 == 16) ? 64 : 128;
}

template <bool FP64>
using ParamsT = typename std::conditional<FP64, Params64, Params32>::type;

template <int D, bool FP64, int N1, class PT>
__device__ __forceinline__ void coeff_scatter_body(const double *__restrict__ q, const double *__restrict__ p,
                                                   const double *__restrict__ s, const double *__restrict__ a,
                                                   int64_t m, int64_t j, const PT &P,
                                                   void *__restrict__ W_v, uint8_t *__restrict__ row_flag,
                                                   int k_first = 0, int k_end = N1) {
    using Real = typename std::conditional<FP64, double, float>::type;
    using C2 = typename std::conditional<FP64, double2, float2>::type;
    constexpr int kT = coeff_threads<FP64, N1>();
    __shared__ C2 scoef[D > 1 ? D - 1 : 1][N1][kT];
    const int tid = threadIdx.x;
    const Common &c = P.c;
    const double ar = a[j], ai = a[m + j];
    if (ar == 0.0 && ai == 0.0) return;  // contributes exact zeros
    // per-dimension coefficients: the last dimension's stay in registers, the
    // others go to this thread's column of shared memory (read back only by
    // this thread, so no barrier is needed)
    Real cl_r[N1], cl_i[N1];
    Real wr, wi;  // weight pref * A * e^{i S/eps} and the packet's gauge phase
    int a0[D], b0[D];
    double rB = 0.0;  // (FP64: that phase, in turns)
    float xy = 0.f;
    // one dimension at a time (for d = 3 not unrolled: three unrolled copies
    // of the coefficient evaluation do not fit the register file)
#pragma unroll(D == 3 ? 1 : D)
    for (int l = 0; l < D; ++l) {
        Real cr[N1], ci[N1];
        if constexpr (FP64) {
            coeff_dim64<N1>(P, q[l * m + j], p[l * m + j], a0[l], b0[l], rB, cr, ci);
        } else {
            float X, Y, zr, zi;
            dim_setup32(c, q[l * m + j], p[l * m + j], a0[l], b0[l], X, Y, zr, zi, rB, xy);
            coeff_dim32<N1>(P, X, Y, zr, zi, 1.f, 0.f, [&](int k, float re, float im) {
                cr[k] = re;
                ci[k] = im;
            });
        }
        if (l < D - 1) {
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                C2 v;
                v.x = cr[k];
                v.y = ci[k];
                scoef[l][k][tid] = v;
            }
        } else {
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                cl_r[k] = cr[k];
                cl_i[k] = ci[k];
            }
        }
    }
    if constexpr (FP64) {
        double ts = s[j] * c.inv_2pi_eps;
        ts -= rint(ts);
        double sn, cs;
        sincospi(2.0 * (ts + rB), &sn, &cs);
        cmul(ar * c.pref, ai * c.pref, cs, sn, wr, wi);
    } else {
        packet_weight32(c, s[j], ar, ai, rB, xy, wr, wi);
    }
    C2 *W = reinterpret_cast<C2 *>(W_v);
    // tensor product over dimensions, innermost dimension last; the rows of
    // the first grid pass (the last dimension's [a][b] plane) that receive a
    // contribution are marked once per row (the single row of d = 1 is marked
    // by the host)
    if constexpr (D == 1) {
        emit_row<D - 1, N1>(W, c, a0[D - 1], b0[D - 1], cl_r, cl_i, 0, wr, wi);
    } else {
#pragma unroll 1
        for (int k0 = k_first; k0 < k_end; ++k0) {  // neighbours of dimension 0
            const int ia0 = a0[0] + c.dq[k0] - c.amin[0], ib0 = b0[0] + c.dp[k0] - c.bmin[0];
            const bool in0 = (unsigned)ia0 < (unsigned)c.A[0] && (unsigned)ib0 < (unsigned)c.B[0];
            if (!in0) continue;
            const int64_t idx0 = ia0 * c.sa[0] + ib0 * c.sb[0];
            const int64_t row0 = ia0 * c.ra[0] + ib0 * c.rb[0];
            const C2 c0 = scoef[0][k0][tid];
            Real p0r, p0i;
            cmul(wr, wi, c0.x, c0.y, p0r, p0i);
            if constexpr (D == 2) {
                row_flag[row0] = 1;
                emit_row<D - 1, N1>(W, c, a0[D - 1], b0[D - 1], cl_r, cl_i, idx0, p0r, p0i);
            } else {
#pragma unroll 1
                for (int k1 = 0; k1 < N1; ++k1) {
                    const int ia1 = a0[1] + c.dq[k1] - c.amin[1], ib1 = b0[1] + c.dp[k1] - c.bmin[1];
                    if ((unsigned)ia1 >= (unsigned)c.A[1] || (unsigned)ib1 >= (unsigned)c.B[1]) continue;
                    const C2 c1 = scoef[1][k1][tid];
                    Real p1r, p1i;
                    cmul(p0r, p0i, c1.x, c1.y, p1r, p1i);
                    row_flag[row0 + ia1 * c.ra[1] + ib1 * c.rb[1]] = 1;
                    emit_row<D - 1, N1>(W, c, a0[D - 1], b0[D - 1], cl_r, cl_i, idx0 + ia1 * c.sa[1] + ib1 * c.sb[1],
                                        p1r, p1i);
                }
            }
        }
    }
}

// d = 1, 2: the compiler's own register budget; d = 3: at most 128
// registers (4 CTAs per SM), which the three-dimensional emit loops need
template <int D, bool FP64, int N1>
__global__ void __launch_bounds__(coeff_threads<FP64, N1>()) coeff_scatter_kernel(
    const double *__restrict__ q, const double *__restrict__ p, const double *__restrict__ s,
    const double *__restrict__ a, int64_t m, const __grid_constant__ ParamsT<FP64> P, void *__restrict__ W_v,
    uint8_t *__restrict__ row_flag) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j < m) coeff_scatter_body<D, FP64, N1>(q, p, s, a, m, j, P, W_v, row_flag);
}

template <int D, bool FP64, int N1>
__global__ void __launch_bounds__(coeff_threads<FP64, N1>(), 4) coeff_scatter3_kernel(
    const double *__restrict__ q, const double *__restrict__ p, const double *__restrict__ s,
    const double *__restrict__ a, int64_t m, const __grid_constant__ ParamsT<FP64> P, void *__restrict__ W_v,
    uint8_t *__restrict__ row_flag) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j < m) coeff_scatter_body<D, FP64, N1>(q, p, s, a, m, j, P, W_v, row_flag);
}

// The same over the packets list[0 .. *count) (device count), grid-stride.  A short
// list takes N1 threads per packet, one neighbour of dimension 0 each (a packet's 512
// reductions one after the other took 46 us of a small 3-D call, 17 us so).
template <int D, bool FP64, int N1>
__global__ void __launch_bounds__(coeff_threads<FP64, N1>(), D == 3 ? 4 : 1) coeff_scatter_list_kernel(
    const double *__restrict__ q, const double *__restrict__ p, const double *__restrict__ s,
    const double *__restrict__ a, int64_t m, const __grid_constant__ ParamsT<FP64> P, void *__restrict__ W_v,
    uint8_t *__restrict__ row_flag, const int *__restrict__ list, const int *__restrict__ count) {
    constexpr int kT = coeff_threads<FP64, N1>();
    const int n = *count;
    const int per = (int64_t)n * N1 <= (int64_t)gridDim.x * kT ? N1 : 1;
    for (int64_t t = blockIdx.x * (int64_t)kT + threadIdx.x; t < (int64_t)n * per; t += (int64_t)gridDim.x * kT) {
        const int k = per == 1 ? 0 : (int)(t % N1);
        coeff_scatter_body<D, FP64, N1>(q, p, s, a, m, list[per == 1 ? t : t / N1], P, W_v, row_flag, k,
                                        per == 1 ? N1 : k + 1);
    }
}

// Batched form: the CTAs of every request of a launch (same dimension,
// precision and neighbour strategy: shared least-squares tables).
template <int D, bool FP64, int N1>
__global__ void __launch_bounds__(coeff_threads<FP64, N1>(), D == 3 ? 4 : 1) coeff_scatter_batch_kernel(
    const __grid_constant__ typename std::conditional<FP64, ScatterBatch64, ScatterBatch32>::type B) {
    int r = 0;
    while (r + 1 < B.n && (int)blockIdx.x >= B.block0[r + 1]) ++r;
    const int64_t j = (int64_t)(blockIdx.x - B.block0[r]) * coeff_threads<FP64, N1>() + threadIdx.x;
    if (j >= B.m[r]) return;
    if constexpr (FP64) {
        const Params64View v{B.c[r], B.f};
        coeff_scatter_body<D, FP64, N1>(B.q[r], B.p[r], B.s[r], B.a[r], B.m[r], j, v, B.W[r], B.flags[r]);
    } else {
        const Params32View v{B.c[r], B.poly};
        coeff_scatter_body<D, FP64, N1>(B.q[r], B.p[r], B.s[r], B.a[r], B.m[r], j, v, B.W[r], B.flags[r]);
    }
}

template <int D>
fgr_status launch_scatter_batch_dim(int n1, cudaStream_t st, const ScatterBatch64 *b64, const ScatterBatch32 *b32) {
    const int nb = b64 ? b64->block0[b64->n] : b32->block0[b32->n];
    if (nb == 0) return FGR_OK;
#define FGR_SB(N)                                                                                      \
    if (b64)                                                                                           \
        coeff_scatter_batch_kernel<D, true, N><<<nb, coeff_threads<true, N>(), 0, st>>>(*b64);         \
    else                                                                                               \
        coeff_scatter_batch_kernel<D, false, N><<<nb, coeff_threads<false, N>(), 0, st>>>(*b32);
    switch (n1) {
    case 4: FGR_SB(4); break;
    case 8: FGR_SB(8); break;
    case 16: FGR_SB(16); break;
    default: set_error("fggc: unsupported neighbour count %d", n1); return FGR_E_INVALID;
    }
#undef FGR_SB
    FGR_CUDA_TRY(cudaGetLastError());
    return FGR_OK;
}

template <int D, bool FP64, int N1>
void launch_coeff_kernel(cudaStream_t st, const PacketsDev &pk, const ParamsT<FP64> &P, void *W, uint8_t *flags) {
    // few packets: smaller CTAs, so that they reach every SM (the FP64 pipe of an
    // SM takes 16 clocks per warp instruction: 4096 packets 66 -> 26 us with the factors below)
    int T = coeff_threads<FP64, N1>();
    while (T > 32 && (pk.m + T - 1) / T < 256) T /= 2;
    const unsigned blocks = (unsigned)((pk.m + T - 1) / T);
    if constexpr (D == 3)
        coeff_scatter3_kernel<D, FP64, N1><<<blocks, T, 0, st>>>(pk.q, pk.p, pk.s, pk.a, pk.m, P, W, flags);
    else
        coeff_scatter_kernel<D, FP64, N1><<<blocks, T, 0, st>>>(pk.q, pk.p, pk.s, pk.a, pk.m, P, W, flags);
}

template <int D>
fgr_status launch_coeff_d(int n1, cudaStream_t st, const PacketsDev &pk, const Params64 *p64, const Params32 *p32,
                          void *W, uint8_t *flags) {
    if (pk.m == 0) return FGR_OK;
#define FGR_COEFF(N)                                                                                        \
    if (p64)                                                                                                \
        launch_coeff_kernel<D, true, N>(st, pk, *p64, W, flags);                                            \
    else                                                                                                    \
        launch_coeff_kernel<D, false, N>(st, pk, *p32, W, flags);
    switch (n1) {
    case 4: FGR_COEFF(4); break;
    case 8: FGR_COEFF(8); break;
    case 16: FGR_COEFF(16); break;
    default: set_error("fggc: unsupported neighbour count %d", n1); return FGR_E_INVALID;
    }
#undef FGR_COEFF
    FGR_CUDA_TRY(cudaGetLastError());
    return FGR_OK;
}

}  // namespace
}  // namespace fgr
