// K2 for d = 1, FP32, on grids that resolve the Gaussian (4 h <= sqrt(eps)).
//
// A thread owns kD1Pts consecutive points.  Around its point x_c a packet's term is
//   term(x_c + k h) = U V^k s^k e^{-(k h)^2 / (2 eps)},
// U the term at x_c, V = e^{i P h / eps} (one per packet) and s = e^{-(x_c - Q) h / eps}
// (real).  The last factor does not depend on the packet, so it multiplies the
// sum at the end; V^k for k = -3 .. 4 is tabulated once per staged packet, with its
// quarter turn beside it, so that each point costs one 16-byte shared load and
// four two-wide instructions (U V^k, the sum, the next power of s).  U takes one
// ex2 and one sine and cosine per thread and packet, and both s and 1/s are
// evaluated, so no power is above the fourth.
// Bound by instruction issue: about 8.5 per packet-point pair, against 17 for four
// points by the recurrences of direct_tile: 1-D workload (262,144 packets, 32,768
// points) 331 -> 259 us with the sum of the slices.  Coarser grids keep direct_tile,
// which has no powers of s across points that lie several widths apart, and so do
// calls with too few packet-point pairs for the partial sums (use_direct1).
// Included by direct.cu inside its anonymous namespace.
#pragma once

constexpr int kD1Threads = 128;
constexpr int kD1Pts = 8;
constexpr int kD1Mid = 3;  // the point with k = 0
static_assert(kD1Threads * kD1Pts == tileT<1>(0), "a CTA owns one tile");

__global__ void __launch_bounds__(kD1Threads) direct1_kernel(const RecF<1> *__restrict__ recs,
                                                             const int64_t *__restrict__ off, const DirectParams P,
                                                             float2 *__restrict__ part) {
    // per staged packet: (window start, length, x - Q at the start, log2 amplitude),
    // V^k and i V^k for k != 0 (at index k + kD1Mid), and the phase constants
    __shared__ __align__(16) float4 sv[kD1Threads][kD1Pts];
    __shared__ __align__(16) float4 sp[kD1Threads];
    const int tid = threadIdx.x, tile = blockIdx.x;
    const int64_t a0 = off[max(0, tile - P.g.K[0])], L = off[tile + 1] - a0;
    const int64_t m0 = (int64_t)tile * tileT<1>(0) + tid * kD1Pts;
    const float mf = (float)m0;
    float2 sum[kD1Pts], low[kD1Pts];  // Kahan sums over the chunks
#pragma unroll
    for (int k = 0; k < kD1Pts; ++k) sum[k] = low[k] = both(0.f);
    // this slice's records: every gridDim.y-th of the list (contiguous shares would
    // differ in how many of their records reach the tile)
    const int64_t n = (L - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y;
    for (int64_t c = 0; c < n; c += kD1Threads) {
        __syncthreads();
        const int nrec = (int)min((int64_t)kD1Threads, n - c);
        if (tid < nrec) {
            const RecF<1> R = recs[a0 + blockIdx.y + (c + tid) * gridDim.y];
            sv[tid][kD1Mid] = make_float4(R.mlo[0], R.wlen[0], R.delta[0], R.la);
            sp[tid] = make_float4(R.nuhi[0], R.nulo[0], R.tau0, 0.f);
#pragma unroll
            for (int k = 1; k <= kD1Pts - 1 - kD1Mid; ++k) {
                float t = (float)k * R.nuhi[0];
                t -= rint_fast(t);
                float sn, cs;
                sincospif(2.f * fmaf((float)k, R.nulo[0], t), &sn, &cs);
                sv[tid][kD1Mid + k] = make_float4(cs, sn, -sn, cs);
                if (k <= kD1Mid) sv[tid][kD1Mid - k] = make_float4(cs, -sn, sn, cs);
            }
        }
        __syncthreads();
        float2 acc[kD1Pts];
#pragma unroll
        for (int k = 0; k < kD1Pts; ++k) acc[k] = both(0.f);
#pragma unroll 1
        for (int j = 0; j < nrec; ++j) {
            const float4 w = sv[j][kD1Mid];
            const float k0 = mf - w.x;  // index in the window of the thread's first point
            if (!(k0 > -(float)kD1Pts && k0 < w.y)) continue;
            const float4 p = sp[j];
            const float kf = k0 + (float)kD1Mid;
            const float dx = fmaf(kf, P.hf[0], w.z);
            float f = kf * p.x;
            f -= rint_fast(f);
            float tau = p.z + fmaf(kf, p.y, f);
            tau -= rint_fast(tau);
            float sn, cs;
            __sincosf(6.283185307179586f * tau, &sn, &cs);
            const float ga = ex2_approx(fmaf(dx * dx, P.ce, w.w));
            const float ds = 2.f * P.ce_h * dx;
            const float2 ur = both(ga * cs), ui = both(ga * sn);
            const float2 up = both(ex2_approx(ds)), dn = both(ex2_approx(-ds));
            auto power = [&](int k, float2 s, bool in) {  // point kD1Mid + k
                const float4 v = sv[j][kD1Mid + k];
                const float2 t = fma2(ui, make_float2(v.z, v.w), mul2(ur, make_float2(v.x, v.y)));
                if (in) acc[kD1Mid + k] = fma2(s, t, acc[kD1Mid + k]);
            };
            const bool whole = k0 >= 0.f && k0 + (float)(kD1Pts - 1) < w.y;
            if (__all_sync(__activemask(), whole)) {
                acc[kD1Mid].x += ur.x;
                acc[kD1Mid].y += ui.x;
                float2 s = up;
#pragma unroll
                for (int k = 1; k <= kD1Pts - 1 - kD1Mid; ++k) {
                    power(k, s, true);
                    s = mul2(s, up);
                }
                s = dn;
#pragma unroll
                for (int k = 1; k <= kD1Mid; ++k) {
                    power(-k, s, true);
                    s = mul2(s, dn);
                }
            } else {
                auto inside = [&](int k) { return kf + (float)k >= 0.f && kf + (float)k < w.y; };
                if (inside(0)) {
                    acc[kD1Mid].x += ur.x;
                    acc[kD1Mid].y += ui.x;
                }
                float2 s = up;
#pragma unroll
                for (int k = 1; k <= kD1Pts - 1 - kD1Mid; ++k) {
                    power(k, s, inside(k));
                    s = mul2(s, up);
                }
                s = dn;
#pragma unroll
                for (int k = 1; k <= kD1Mid; ++k) {
                    power(-k, s, inside(-k));
                    s = mul2(s, dn);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kD1Pts; ++k) {
            kahan_sum(sum[k].x, low[k].x, acc[k].x);
            kahan_sum(sum[k].y, low[k].y, acc[k].y);
        }
    }
    // the slice's share of the tile (direct1_sum_kernel adds the slices)
    float2 *to = part + (int64_t)blockIdx.y * gridDim.x * tileT<1>(0) + m0;
#pragma unroll
    for (int k = 0; k < kD1Pts; k += 2) {
        float4 v;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float d = (float)(k + h - kD1Mid) * P.hf[0], e = ex2_approx(d * d * P.ce);
            (h ? v.z : v.x) = e * (sum[k + h].x - low[k + h].x);
            (h ? v.w : v.y) = e * (sum[k + h].y - low[k + h].y);
        }
        *reinterpret_cast<float4 *>(to + k) = v;
    }
}

// u[m] = the sum of the slices (compensated): a store and a read per slice cost what
// an atomic would, and neither their order nor their number touches the result's
// precision.
// A CTA takes 32 points; its eight warps share out the slices.
__global__ void __launch_bounds__(256) direct1_sum_kernel(const float2 *__restrict__ part, int slices, int64_t stride,
                                                          int64_t n, float2 *__restrict__ u) {
    __shared__ float4 sub[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t m = blockIdx.x * (int64_t)32 + lane;
    float2 s = both(0.f), c = both(0.f);
#pragma unroll 4
    for (int y = w; y < slices; y += 8) {
        const float2 v = part[y * stride + m];  // (the stride covers whole tiles)
        kahan_sum(s.x, c.x, v.x);
        kahan_sum(s.y, c.y, v.y);
    }
    sub[w][lane] = make_float4(s.x, s.y, c.x, c.y);
    __syncthreads();
    if (w > 0 || m >= n) return;
#pragma unroll
    for (int i = 1; i < 8; ++i) {
        const float4 v = sub[i][lane];
        c.x += v.z;
        c.y += v.w;
        kahan_sum(s.x, c.x, v.x);
        kahan_sum(s.y, c.y, v.y);
    }
    u[m] = make_float2(s.x - c.x, s.y - c.y);
}
