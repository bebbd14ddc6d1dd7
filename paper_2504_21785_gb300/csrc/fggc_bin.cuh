// K4 for d = 2, 3 (FP32 path): the scatter of eq. 2.25 with the packets binned
// by anchor cell.
//
// A packet's contributions to one row of the node array (the last dimension's
// [a][b] plane for fixed outer nodes) are the neighbours of its inner anchor
// cell, and the outer anchor cell (a0, b0 of the other dimensions) fixes which
// n1^(d-1) rows it reaches.  Packets with the same outer anchor cell (d = 2: and
// the same 24 x 16 tile of inner anchors, so that they overlap) form a bin.
// After a counting sort by bin a CTA takes up to kBinT packets of one, lists for
// every target cell of their inner box the (packet, neighbour) pairs that reach
// it, sums a cell's contributions to every row in registers and adds each row's
// value to W with one 8-byte reduction: one per touched (cell, row) instead of
// one per contribution, issued by neighbouring lanes to neighbouring cells.  A
// packet set of one packet per dq x dp cell (what the flow preserves) gives 6
// to 8 pairs per cell.
//
// The sort's last kernel also turns each packet into a 48-byte record in bin
// order (cell offsets, weight and phases: all that needs more than FP32), so
// that the binned kernel reads its packets in one piece and does FP32 work only.
// Bins with fewer than kBinMinCount packets go through the per-packet kernel
// (fggc_coeff.cuh) from a list.
//
// Included by fggc_coeff2.cu and fggc_coeff3.cu.
#pragma once

#include <algorithm>
#include <climits>

#include "fggc_coeff.cuh"

namespace fgr {
namespace {

constexpr int kBinT = 256;         // packets (threads) per binned item
// Resident binned-scatter CTAs per SM (registers; d = 3: and shared memory).
template <int D>
__host__ __device__ constexpr int bin_ctas_per_sm() {
    return D == 3 ? 3 : 4;
}

// Warp-aggregated atomicAdd of 1 on ctr[k] by the active lanes (one atomic per
// distinct k); returns the old value plus the lane's rank among the lanes with
// the same k.
__device__ __forceinline__ int aggregated_add(int *ctr, int k) {
    const unsigned act = __activemask();
    const unsigned peers = __match_any_sync(act, k);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    const int rank = __popc(peers & ((1u << lane) - 1));
    int base = 0;
    if (lane == leader) base = atomicAdd(ctr + k, __popc(peers));
    base = __shfl_sync(peers, base, leader);
    return base + rank;
}

// Per packet: its key (-1: the packet adds nothing: zero amplitude, or every
// node of a keyed dimension lies outside the node box) and its place among the
// packets of that key, counted in count[].
template <int D>
__global__ void __launch_bounds__(256) bin_key_kernel(const double *__restrict__ q, const double *__restrict__ p,
                                                      const double *__restrict__ a, int64_t m, const Common c,
                                                      const BinBox bb, int *__restrict__ key, int *__restrict__ rank,
                                                      int *__restrict__ count) {
    constexpr int KD = D == 2 ? 2 : D - 1;  // dimensions that the key reads
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= m) return;
    int k = -1;
    double qv[KD], pv[KD];  // every load first (none waits on the amplitude test)
#pragma unroll
    for (int l = 0; l < KD; ++l) {
        qv[l] = q[l * m + j];
        pv[l] = p[l * m + j];
    }
    if (a[j] != 0.0 || a[m + j] != 0.0) {
        int64_t kk = 0;
        bool ok = true;
#pragma unroll
        for (int l = 0; l < KD; ++l) {
            int ia = floor_div_int(qv[l], c.dqv, c.inv_dq) - bb.ka_lo[l];
            int ib = floor_div_int(pv[l], c.dpv, c.inv_dp) - bb.kb_lo[l];
            ok = ok && (unsigned)ia < (unsigned)bb.KA[l] && (unsigned)ib < (unsigned)bb.KB[l];
            const bool inner = l == D - 1;
            kk = (kk * (inner ? bb.tiles_a : bb.KA[l]) + (inner ? (unsigned)ia / kBinTileA : ia)) *
                     (inner ? bb.tiles_b : bb.KB[l]) +
                 (inner ? (unsigned)ib / kBinTileB : ib);
        }
        if (ok) k = (int)kk;
    }
    key[j] = k;
    if (k >= 0) rank[j] = aggregated_add(count, k);
}

// x / step of a packet coordinate as integer part fl and offset fr in [0, 1),
// with the quotient p + e (FP32 sum, relative error below 2^-45); within 2^-20 of
// an integer the FP64 division decides the integer part.  False: out of the
// range in which offsets and phases keep FP32 accuracy (the caller's FP64 path).
__device__ __forceinline__ bool quotient_split(double x, const float *inv, double step, double inv_step, float &fl,
                                               float &fr, float &p, float &e) {
    float h, l;
    bool ok = split_double(x, h, l);
    p = __fmul_rn(h, inv[0]);
    e = fmaf(h, inv[0], -p);
    e = fmaf(h, inv[1], e);
    e = fmaf(l, inv[0], e);
    ok = ok && fabsf(p) < 262144.f;
    fl = floorf(p);
    fr = __fadd_rn(__fsub_rn(p, fl), e);
    if (fr < 0.f) {
        fl -= 1.f;
        fr += 1.f;
    } else if (fr >= 1.f) {
        fl += 1.f;
        fr -= 1.f;
    }
    if (ok && (fr < 0x1p-20f || fr > 1.f - 0x1p-20f)) {
        const float f = (float)floor(quotient_for_floor(x, step, inv_step));
        fr += fl - f;
        fl = f;
    }
    return ok;
}

// (p + e) k in turns: t the part reduced to [-1/2, 1/2], returned, lo the rest.
__device__ __forceinline__ float turns_split(float p, float e, const float *k, float &lo) {
    const float t = __fmul_rn(p, k[0]);
    float u = fmaf(p, k[0], -t);
    u = fmaf(p, k[1], u);
    lo = fmaf(e, k[0], u);
    return __fsub_rn(t, rint_fast(t));
}

// s += x (error-free, the rounding goes to lo), reduced to [-1/2, 1/2].
__device__ __forceinline__ void turns_add(float &s, float &lo, float x) {
    const float v = __fadd_rn(s, x), b = __fsub_rn(v, s);
    lo += __fadd_rn(__fsub_rn(s, __fsub_rn(v, b)), __fsub_rn(x, b));
    s = __fsub_rn(v, rint_fast(v));
}

// A packet's record: offsets (sx, ty) per dimension, weight, z of the last
// dimension and its anchor (see dim_setup32 and packet_weight32, whose FP64
// phases these are).  FP64 instructions take 16 clocks of an SM here, so the
// offsets and phases are computed as FP32 sums (2^-45 relative); packets out of
// range (|Q/dq| or |P/dp| >= 2^18, |S| / (2 pi eps) >= 2^18 turns, amplitudes
// below 2^-100) take the FP64 form.
template <int D>
__device__ __forceinline__ void packet_record(const Common &c, const SplitConst &k, const double *qv,
                                              const double *pv, double s, double ar, double ai, float *sx, float *ty,
                                              int &a0, int &b0, float2 &w, float2 &z) {
    bool ok = true;
    float h, l, xy = 0.f, T, lo;
    ok = split_double(s, h, l) && ok;
    ok = ok && fabsf(h * k.inv_2pi_eps[0]) < 262144.f;
    T = turns_split(h, l, k.inv_2pi_eps, lo);
    float A = 0.f;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        float fa, fb, fr, p, e, pb, eb;
        ok = quotient_split(pv[d], k.inv_dp, c.dpv, c.inv_dp, fb, fr, pb, eb) && ok;
        ty[d] = fr - 0.5f;
        ok = quotient_split(qv[d], k.inv_dq, c.dqv, c.inv_dq, fa, fr, p, e) && ok;
        sx[d] = fr - 0.5f;
        const float B = fb + 0.5f, g = __fmul_rn(p, B);
        ok = ok && fabsf(g * k.cc[0]) < 262144.f;
        float u;
        const float t = turns_split(g, fmaf(e, B, fmaf(p, B, -g)), k.cc, u);
        turns_add(T, lo, -t);
        lo -= u;
        xy = fmaf(sx[d], ty[d], xy);
        if (d == D - 1) {
            a0 = (int)fa;
            b0 = (int)fb;
            A = fa + 0.5f;
        }
    }
    float sn, cs;
    if (ok) {
        sincospif(2.f * (T + fmaf(-0.5f * k.cc[0], xy, lo)), &sn, &cs);
        ok = split_double(ar, h, l);
        const float wr = fmaf(h, k.pref[0], fmaf(h, k.pref[1], l * k.pref[0]));
        ok = split_double(ai, h, l) && ok;
        const float wi = fmaf(h, k.pref[0], fmaf(h, k.pref[1], l * k.pref[0]));
        cmul(wr, wi, cs, sn, w.x, w.y);
        float u;
        const float t = turns_split(A, 0.f, k.half_cc, u);
        sincospif(2.f * (t + u), &z.y, &z.x);
    }
    if (!ok) {
        double rB = 0.0;
        xy = 0.f;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            float X, Y;
            dim_setup32(c, qv[d], pv[d], a0, b0, X, Y, z.x, z.y, rB, xy);
            sx[d] = 0.5f * X;
            ty[d] = 0.5f * Y;
        }
        packet_weight32(c, s, ar, ai, rB, xy, w.x, w.y);
    }
}

// Writes every binned packet's record at its place (and, d = 3, widens the inner
// anchor box of its key) and puts every packet of a small bin on the loose list.
template <int D>
__global__ void __launch_bounds__(256) bin_place_kernel(const double *__restrict__ q, const double *__restrict__ p,
                                                        const double *__restrict__ s, const double *__restrict__ a,
                                                        int64_t m, const __grid_constant__ Common c,
                                                        const __grid_constant__ SplitConst sc,
                                                        const int *__restrict__ key, const int *__restrict__ rank,
                                                        const int2 *__restrict__ off, BinRecord *__restrict__ rec,
                                                        int4 *kbox, int *__restrict__ loose, int *__restrict__ nloose) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= m) return;
    const int k = key[j];
    double qv[D], pv[D];
#pragma unroll
    for (int l = 0; l < D; ++l) {
        qv[l] = q[l * m + j];
        pv[l] = p[l * m + j];
    }
    const double sv = s[j], ar = a[j], ai = a[m + j];
    if (k < 0) return;
    const int2 o = off[k], o1 = off[k + 1];
    int a0, b0;
    if (o1.x == o.x) {
        loose[aggregated_add(nloose, 0)] = (int)j;
        a0 = floor_div_int(qv[D - 1], c.dqv, c.inv_dq) - c.amin[D - 1];
        b0 = floor_div_int(pv[D - 1], c.dpv, c.inv_dp) - c.bmin[D - 1];
    } else {
        float sx[D], ty[D];
        float2 w, z;
        packet_record<D>(c, sc, qv, pv, sv, ar, ai, sx, ty, a0, b0, w, z);
        a0 -= c.amin[D - 1];
        b0 -= c.bmin[D - 1];
        BinRecord r;
        r.x = make_float4(sx[0], ty[0], sx[D - 1], ty[D - 1]);
        r.w = make_float4(w.x, w.y, z.x, z.y);
        r.y = make_float4(__int_as_float(a0), __int_as_float(b0), sx[D / 2], ty[D / 2]);
        rec[o.x + rank[j]] = r;
    }
    if constexpr (D == 3) {
        // most packets find their key's box wide enough already (a stale read
        // only costs an atomic)
        const int4 b = __ldcg(kbox + k);
        int *kb = reinterpret_cast<int *>(kbox + k);
        if (a0 < b.x) atomicMin(kb, a0);
        if (-a0 < b.y) atomicMin(kb + 1, -a0);
        if (b0 < b.z) atomicMin(kb + 2, b0);
        if (-b0 < b.w) atomicMin(kb + 3, -b0);
    }
}

// Outer anchors of a key (and the tile index of its inner anchors).
template <int D>
__device__ __forceinline__ void key_anchors(const BinBox &bb, unsigned k, int *oa, int *ob, int &ta, int &tb) {
    tb = 0;
    ta = 0;
    if (D == 2) {
        tb = (int)(k % (unsigned)bb.tiles_b);
        k /= (unsigned)bb.tiles_b;
        ta = (int)(k % (unsigned)bb.tiles_a);
        k /= (unsigned)bb.tiles_a;
    }
#pragma unroll
    for (int l = D - 2; l >= 0; --l) {
        ob[l] = (int)(k % (unsigned)bb.KB[l]) + bb.kb_lo[l];
        k /= (unsigned)bb.KB[l];
        oa[l] = (int)(k % (unsigned)bb.KA[l]) + bb.ka_lo[l];
        k /= (unsigned)bb.KA[l];
    }
}

// Inner target box (ta0, ta1, tb0, tb1) of a key's packets in the node box;
// false if their neighbours reach past the node box.
template <int D>
__device__ __forceinline__ bool key_box(const Common &c, const BinBox &bb, const int4 *kbox, int64_t k, int ta, int tb,
                                        int4 &box) {
    int4 an;  // inner anchors: first and last a, first and last b (relative to the node box)
    if constexpr (D == 3) {
        const int4 b = kbox[k];
        an = make_int4(b.x, -b.y, b.z, -b.w);
    } else {
        an.x = bb.ka_lo[1] - c.amin[1] + ta * kBinTileA;
        an.y = bb.ka_lo[1] - c.amin[1] + min(bb.KA[1], (ta + 1) * kBinTileA) - 1;
        an.z = bb.kb_lo[1] - c.bmin[1] + tb * kBinTileB;
        an.w = bb.kb_lo[1] - c.bmin[1] + min(bb.KB[1], (tb + 1) * kBinTileB) - 1;
    }
    an.x += bb.dqmin;
    an.y += bb.dqmax;
    an.z += bb.dpmin;
    an.w += bb.dpmax;
    box = make_int4(max(0, an.x), min(c.A[D - 1] - 1, an.y), max(0, an.z), min(c.B[D - 1] - 1, an.w));
    return an.x >= 0 && an.y < c.A[D - 1] && an.z >= 0 && an.w < c.B[D - 1];
}

// One item per kBinT packets of every bin.
template <int D>
__global__ void bin_items_kernel(const int2 *__restrict__ off, const int4 *__restrict__ kbox, const Common c,
                                 const BinBox bb, BinItem *__restrict__ items) {
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= bb.K) return;
    const int2 o = off[k], o1 = off[k + 1];
    const int n = o1.x - o.x;
    if (n == 0) return;
    int oa[D - 1], ob[D - 1], ta, tb;
    key_anchors<D>(bb, (unsigned)k, oa, ob, ta, tb);
    BinItem it;
    const bool inside = key_box<D>(c, bb, kbox, k, ta, tb, it.box);
    float z[4] = {1.f, 0.f, 1.f, 0.f};
#pragma unroll
    for (int l = 0; l < D - 1; ++l) {
        double t = 0.5 * c.cc * ((double)oa[l] + 0.5);
        t -= rint(t);
        sincospif(2.f * (float)t, &z[2 * l + 1], &z[2 * l]);
    }
    it.z = make_float4(z[0], z[1], z[2], z[3]);
    for (int t = 0; t < o1.y - o.y; ++t) {
        it.at = make_int4((int)k, o.x + t * kBinT, min(kBinT, n - t * kBinT), inside ? 1 : 0);
        items[o.y + t] = it;
    }
}

// Before the scatter: marks every row of W that the packets of an occupied key
// will reach (the n1^(d-1) outer neighbours of its anchor cell that lie in the
// node box) and widens the rows' boxes (min a, min -a, min b, min -b of the inner
// nodes; d = 2: min a, min -a per four b values) by the key's.  per (1 or 8) threads per key share out the neighbours of
// dimension 0: eight where the keys are few (90,000 of them 29 -> 15 us), one where
// most threads would only find an empty key (888,000: 43 us against 62).  The binned
// and per-packet kernels
// reach exactly these rows, so only they need clearing.
template <int D>
__global__ void bin_mark_rows_kernel(const int *__restrict__ count, const int4 *__restrict__ kbox, const Common c,
                                     const BinBox bb, int per, uint8_t *__restrict__ row_flag, int4 *row_box,
                                     int2 *row_range, int halves) {
    const int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) / per;
    if (k >= bb.K || count[k] == 0) return;
    int oa[D - 1], ob[D - 1], ta, tb;
    key_anchors<D>(bb, (unsigned)k, oa, ob, ta, tb);
    int4 box;
    key_box<D>(c, bb, kbox, k, ta, tb, box);
    const bool lands = box.x <= box.y && box.z <= box.w;
    auto mark = [&](int64_t row) {
        row_flag[row] = 1;
        if (!lands) return;
        // (a stale read only costs an atomic)
        if constexpr (D == 2) {
            for (int h = box.z / kRowHalf; h <= box.w / kRowHalf; ++h) {
                int2 *x = row_range + row * halves + h;
                const int2 now = __ldcg(x);
                if (box.x < now.x) atomicMin(&x->x, box.x);
                if (-box.y < now.y) atomicMin(&x->y, -box.y);
            }
            return;
        }
        const int4 v = __ldcg(row_box + row);
        int *b = reinterpret_cast<int *>(row_box + row);
        if (box.x < v.x) atomicMin(b, box.x);
        if (-box.y < v.y) atomicMin(b + 1, -box.y);
        if (box.z < v.z) atomicMin(b + 2, box.z);
        if (-box.w < v.w) atomicMin(b + 3, -box.w);
    };
    for (int k0 = threadIdx.x % per; k0 < c.n1; k0 += per) {
        const int ia0 = oa[0] + c.dq[k0] - c.amin[0], ib0 = ob[0] + c.dp[k0] - c.bmin[0];
        if ((unsigned)ia0 >= (unsigned)c.A[0] || (unsigned)ib0 >= (unsigned)c.B[0]) continue;
        const int64_t row0 = (int64_t)ia0 * c.ra[0] + (int64_t)ib0 * c.rb[0];
        if constexpr (D == 2) {
            mark(row0);
        } else {
            for (int k1 = 0; k1 < c.n1; ++k1) {
                const int ia1 = oa[1] + c.dq[k1] - c.amin[1], ib1 = ob[1] + c.dp[k1] - c.bmin[1];
                if ((unsigned)ia1 >= (unsigned)c.A[1] || (unsigned)ib1 >= (unsigned)c.B[1]) continue;
                mark(row0 + (int64_t)ia1 * c.ra[1] + (int64_t)ib1 * c.rb[1]);
            }
        }
    }
}

// Zeroes the flagged rows of W (row_f4 16-byte words each): a warp reads the
// flags of 32 consecutive rows at once and clears its part (blockIdx.y of
// gridDim.y) of the flagged ones together.
__global__ void __launch_bounds__(256) clear_flagged_rows_kernel(float4 *__restrict__ W,
                                                                 const uint8_t *__restrict__ row_flag,
                                                                 int64_t rows, int64_t row_f4) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t base = (blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5)) * 32; base < rows;
         base += nwarps * 32) {
        const bool f = base + lane < rows && row_flag[base + lane] != 0;
        unsigned set = __ballot_sync(0xffffffffu, f);
        const int64_t part = (row_f4 + gridDim.y - 1) / gridDim.y, i0 = blockIdx.y * part;
        const int64_t i1 = min(row_f4, i0 + part);
        while (set) {
            const int r = __ffs(set) - 1;
            set &= set - 1;
            float4 *p = W + (base + r) * row_f4;
            for (int64_t i = i0 + lane; i < i1; i += 32) p[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
    }
}

// Target cells of one window (node cells of the inner plane).
constexpr int kWinCells = 1024;

// float2 slots per packet in the coefficient array: D x N1 rounded to an odd
// number of 16-byte words, so that the 16-byte loads of different packets by
// the lanes of a warp spread over all bank groups instead of two
template <int D, int N1>
__host__ __device__ constexpr int coef_stride() {
    return D * N1 + (((D * N1 / 2) % 2 == 0) ? 2 : 0);
}

template <int D, int N1>
__host__ __device__ constexpr int binned_smem_bytes() {
    return kBinT * coef_stride<D, N1>() * 8  // coefficients [packet][dimension][neighbour] (float2)
           + kWinCells * 4         // entries per cell (int)
           + kWinCells * 4         // per cell: first entry, end of its entries (16 bits each)
           + kWinCells * 4         // active cells (packed line, column)
           + (D == 3 ? N1 * N1 : N1) * 8  // W offsets of the rows (int64)
           + kBinT * N1 * 2;       // entries (packet << 4 | neighbour), uint16
}

// Binned coefficient + scatter: persistent CTAs take items from *work.  All
// packets of an item share the outer anchor cell, so they reach the same
// n1^(d-1) rows, and a target cell of the inner plane receives, in every row,
// the sum over its entries (packet j, inner neighbour k) of
//   w_j c_{d-1,j}[k] * c_{0,j}[k0] (* c_{1,j}[k1]).
// Per item (and window of whole inner q-node lines of the target box) the CTA
// lists every target cell's entries (a CSR built once); then NP lanes per cell
// accumulate its rows in registers as a sum of outer products over its entries
// and add each row's value to W with one 8-byte reduction.  No floating-point
// atomics in shared memory.
// Bound by the shared-memory pipe and the barriers between the phases of an item
// (2-D workload: data pipe 66 %, issue 59 %; 3-D, 2M packets: 74 %, 50 %).  3-D workload
// (16.8M packets): 7.45 -> 5.73 ms with the FP64 part and the packet gathers in
// the sort (whose last kernel grew from 0.09 to 0.76 ms), 2-D (4.2M): 1.02 ms
// per packet -> 0.50 ms.
template <int D, int N1>
__global__ void __launch_bounds__(kBinT, bin_ctas_per_sm<D>()) binned_scatter_kernel(
    const __grid_constant__ Params32 P, const __grid_constant__ BinBox bb, const BinRecord *__restrict__ rec,
    const BinItem *__restrict__ items, const int2 *__restrict__ off_end, int *__restrict__ work,
    float2 *__restrict__ W) {
    constexpr int NR = D == 3 ? N1 * N1 : N1;       // rows reached by one outer anchor cell
    constexpr int NP = D == 3 && N1 == 8 ? 4 : 1;   // lanes per target cell
    constexpr int NA = N1 / NP;                     // k0 values per lane
    constexpr int NK1 = D == 3 ? N1 : 2;            // k1 values (d = 2: none)
    constexpr int kSub = 32 / NP;                   // target cells per warp
    constexpr int kPer = kWinCells / kBinT;         // target cells per thread in the CSR build
    constexpr int CS = coef_stride<D, N1>();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // [kBinT][CS] per packet: pairs of neighbours as (re, re', im, im') for the
    // outer dimensions (the operands of the packed multiply-adds), (re, im) times
    // the packet's weight for the last; padding
    float2 *coef = reinterpret_cast<float2 *>(smem_raw);
    int *cnt = reinterpret_cast<int *>(coef + kBinT * CS);             // [kWinCells], zero between windows
    unsigned *span = reinterpret_cast<unsigned *>(cnt + kWinCells);    // [kWinCells]
    unsigned *act = span + kWinCells;                                  // [kWinCells]
    int64_t *rowoff = reinterpret_cast<int64_t *>(act + kWinCells);    // [NR]
    unsigned short *ent = reinterpret_cast<unsigned short *>(rowoff + NR);  // [kBinT * N1]
    __shared__ __align__(16) BinItem s_item[2];
    __shared__ unsigned s_rows[2];  // bit r: row r lies in the node box
    __shared__ int2 s_sum[kBinT / 32];
    const Common &c = P.c;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int nitems = off_end->y;
    // thread 0 fetches the next item (asynchronous copies into shared memory)
    // while the CTA works on the current one
    auto fetch = [&](BinItem *to, int i) {
        if (i < nitems) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(to);
#pragma unroll
            for (int o = 0; o < (int)sizeof(BinItem); o += 16)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + o),
                             "l"(reinterpret_cast<const char *>(items + i) + o)
                             : "memory");
        } else {
            to->at = make_int4(0, 0, 0, 0);
        }
    };
    auto fetched = [] { asm volatile("cp.async.wait_all;" ::: "memory"); };
    if (tid == 0) {
        fetch(&s_item[0], atomicAdd(work, 1));
        fetched();
    }
    if (tid < 2) s_rows[tid] = 0u;
    for (int e = tid; e < kWinCells; e += kBinT) cnt[e] = 0;
    for (int buf = 0;; buf ^= 1) {
        __syncthreads();  // the item is there; the previous one's shared data are no longer read
        const int4 at = s_item[buf].at, box = s_item[buf].box;
        if (at.z == 0) break;
        int next = 0;
        if (tid == 0) next = atomicAdd(work, 1);
        const bool valid = tid < at.z;
        const int ta0 = box.x, tb0 = box.z, TA = box.y - ta0 + 1, TB = box.w - tb0 + 1;
        const int WH = TA > 0 && TB > 0 ? kWinCells / TB : 0;  // inner q-node lines per window
        float2 *cj = coef + tid * CS;
        int ra = 0, rb = 0;  // inner anchor relative to the node box
        // the packet's target cells in the window of lines [wa, wa + wn), without
        // tests when the whole box is one window inside the node box
        const bool plain = at.w != 0 && TA <= WH;
        auto each_entry = [&](int wa, int wn, auto f) {
            if (plain) {
                const int e = (ra - ta0) * TB + rb - tb0;
#pragma unroll
                for (int k = 0; k < N1; ++k) f(k, e + c.dq[k] * TB + c.dp[k]);
            } else {
#pragma unroll
                for (int k = 0; k < N1; ++k) {
                    const int ia = ra + c.dq[k] - ta0 - wa, ib = rb + c.dp[k] - tb0;
                    if ((unsigned)ia < (unsigned)wn && (unsigned)ib < (unsigned)TB) f(k, ia * TB + ib);
                }
            }
        };
        if (valid) {
            const BinRecord *r = rec + at.y + tid;
            const float4 x = r->x, w = r->w, y = r->y, z = s_item[buf].z;
            ra = __float_as_int(y.x);
            rb = __float_as_int(y.y);
            if (WH > 0) each_entry(0, min(WH, TA), [&](int, int e) { atomicAdd(&cnt[e], 1); });
            // one dimension at a time (one copy of the evaluation: two would keep
            // its constants in registers)
#pragma unroll 1
            for (int l = 0; l < D; ++l) {
                const bool last = l == D - 1;
                float *cl = reinterpret_cast<float *>(cj + l * N1);
                coeff_dim32<N1>(P, 2.f * (last ? x.z : l == 0 ? x.x : y.z), 2.f * (last ? x.w : l == 0 ? x.y : y.w),
                                last ? w.z : l == 0 ? z.x : z.z, last ? w.w : l == 0 ? z.y : z.w,
                                last ? w.x : 1.f, last ? w.y : 0.f, [&](int k, float re, float im) {
                                    const int b = 4 * (k >> 1) + (k & 1);
                                    cl[last ? 2 * k : b] = re;
                                    cl[last ? 2 * k + 1 : b + 2] = im;
                                });
            }
        }
        // the rows of the item's outer anchor cell: W offsets and in-box bits
        if (tid < (NR + 31) / 32 * 32) {
            bool in = tid < NR;
            if (in) {
                int oa[D - 1], ob[D - 1], ta, tb;
                key_anchors<D>(bb, (unsigned)at.x, oa, ob, ta, tb);
                const int k0 = D == 3 ? tid / N1 : tid, k1 = D == 3 ? tid % N1 : 0;
                const int ia0 = oa[0] + c.dq[k0] - c.amin[0], ib0 = ob[0] + c.dp[k0] - c.bmin[0];
                in = (unsigned)ia0 < (unsigned)c.A[0] && (unsigned)ib0 < (unsigned)c.B[0];
                int64_t idx = (int64_t)ia0 * c.sa[0] + (int64_t)ib0 * c.sb[0];
                if constexpr (D == 3) {
                    const int ia1 = oa[1] + c.dq[k1] - c.amin[1], ib1 = ob[1] + c.dp[k1] - c.bmin[1];
                    in = in && (unsigned)ia1 < (unsigned)c.A[1] && (unsigned)ib1 < (unsigned)c.B[1];
                    idx += (int64_t)ia1 * c.sa[1] + (int64_t)ib1 * c.sb[1];
                }
                rowoff[tid] = idx;
            }
            const unsigned bits = __ballot_sync(0xffffffffu, in);
            if (lane == 0) s_rows[wid] = bits;
        }
        __syncthreads();
        if (tid == 0) fetch(&s_item[buf ^ 1], next);
        const unsigned long long rows_in = s_rows[0] | (unsigned long long)s_rows[1] << 32;
        if (TA > 0 && TB > 0 && WH == 0 && valid) {
            // a b-range wider than a window: one reduction per contribution
            float cr[N1], ci[N1];
#pragma unroll
            for (int k = 0; k < N1; ++k) {
                const float2 v = cj[(D - 1) * N1 + k];
                cr[k] = v.x;
                ci[k] = v.y;
            }
#pragma unroll 1
            for (int r = 0; r < NR; ++r) {
                if (!((rows_in >> r) & 1ull)) continue;
                const int k0 = D == 3 ? r / N1 : r, k1 = D == 3 ? r % N1 : 0;
                const float *c0 = reinterpret_cast<const float *>(cj) + 4 * (k0 >> 1) + (k0 & 1);
                float pr = c0[0], pi = c0[2];  // the weight is in cr, ci
                if constexpr (D == 3) {
                    const float *c1 = reinterpret_cast<const float *>(cj + N1) + 4 * (k1 >> 1) + (k1 & 1);
                    float tr, ti;
                    cmul(pr, pi, c1[0], c1[2], tr, ti);
                    pr = tr;
                    pi = ti;
                }
                emit_row<D - 1, N1>(W, c, ra + c.amin[D - 1], rb + c.bmin[D - 1], cr, ci, rowoff[r], pr, pi);
            }
        }
        const int nwin = WH > 0 && rows_in != 0ull ? (TA + WH - 1) / WH : 0;
        if (nwin == 0 && WH > 0)  // nothing lands in the node box: drop the counts
            for (int e = tid; e < kWinCells; e += kBinT) cnt[e] = 0;
#pragma unroll 1
        for (int w = 0; w < nwin; ++w) {
            const int wa = w * WH, wn = min(WH, TA - wa), cells = wn * TB;
            if (w > 0) {
                __syncthreads();  // the previous window's lists are no longer read
                if (valid) each_entry(wa, wn, [&](int, int e) { atomicAdd(&cnt[e], 1); });
                __syncthreads();
            }
            // --- entry starts and the ordered list of non-empty cells by one block
            // scan over the counts (thread t: cells [t kPer, (t + 1) kPer)) --------
            int nact;
            {
                int n[kPer];
                int2 loc = make_int2(0, 0);
                const int4 v = *reinterpret_cast<const int4 *>(cnt + tid * kPer);
                static_assert(kPer == 4, "one 16-byte load of counts per thread");
                n[0] = v.x;
                n[1] = v.y;
                n[2] = v.z;
                n[3] = v.w;
                *reinterpret_cast<int4 *>(cnt + tid * kPer) = make_int4(0, 0, 0, 0);
#pragma unroll
                for (int i = 0; i < kPer; ++i) {
                    loc.x += n[i];
                    loc.y += n[i] > 0;
                }
                int2 inc = loc;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int ux = __shfl_up_sync(0xffffffffu, inc.x, o), uy = __shfl_up_sync(0xffffffffu, inc.y, o);
                    if (lane >= o) {
                        inc.x += ux;
                        inc.y += uy;
                    }
                }
                if (lane == 31) s_sum[wid] = inc;
                __syncthreads();
                int2 base = make_int2(inc.x - loc.x, inc.y - loc.y);
                nact = 0;
#pragma unroll
                for (int i = 0; i < kBinT / 32; ++i) {
                    const int2 v2 = s_sum[i];
                    if (i < wid) {
                        base.x += v2.x;
                        base.y += v2.y;
                    }
                    nact += v2.y;
                }
#pragma unroll
                for (int i = 0; i < kPer; ++i) {
                    const int e = tid * kPer + i;
                    if (e < cells) {
                        span[e] = (unsigned)base.x * 0x10001u;  // first entry, cursor of the fill below
                        if (n[i] > 0) {
                            const int ia = e / TB, ib = e - ia * TB;
                            act[base.y++] = ((unsigned)ia << 16) | (unsigned)ib;
                        }
                        base.x += n[i];
                    }
                }
            }
            __syncthreads();
            if (valid)
                each_entry(wa, wn, [&](int k, int e) {
                    ent[atomicAdd(&span[e], 0x10000u) >> 16] = (unsigned short)((tid << 4) | k);
                });
            __syncthreads();
            // --- cells: rows in registers, then one reduction per row ----------
            // A warp takes kSub consecutive cells; its NP lanes per cell share out
            // the k0 values, so they walk the same entries and a warp waits for
            // the longest of kSub lists instead of 32.
            const int kp = lane % NP;
            for (int g0 = wid * kSub; g0 < nact; g0 += kBinT / 32 * kSub) {
                const int i = g0 + lane / NP;
                if (i >= nact) continue;
                const unsigned cell = act[i];
                const int ia = (int)(cell >> 16), ib = (int)(cell & 0xffffu);
                const unsigned sp = span[ia * TB + ib];
                const int x0 = (int)(sp & 0xffffu), x1 = (int)(sp >> 16);
                float2 *Wc = W + (int64_t)(ta0 + wa + ia) * c.sa[D - 1] + tb0 + ib;
                // pairs of k1 (d = 3) or of k0 (d = 2)
                constexpr int NU = D == 3 ? NA : 1, NV = D == 3 ? NK1 / 2 : NA / 2;
                float2 accr[NU][NV], acci[NU][NV];
#pragma unroll
                for (int u = 0; u < NU; ++u)
#pragma unroll
                    for (int v = 0; v < NV; ++v) accr[u][v] = acci[u][v] = both(0.f);
                for (int xe = x0; xe < x1; ++xe) {
                    const int en = ent[xe], jj = en >> 4, kk = en & 15;
                    const float2 ev = coef[jj * CS + (D - 1) * N1 + kk];  // w c_{d-1}[k]
                    const float4 *cp4 = reinterpret_cast<const float4 *>(coef + jj * CS);
                    float2 tr[NA / 2], ti[NA / 2];  // pairs of k0 (d = 3)
                    if constexpr (D == 3) {
#pragma unroll
                        for (int u = 0; u < NA / 2; ++u) {
                            const float4 t = cp4[kp * (NA / 2) + u];
                            const float2 re = make_float2(t.x, t.y), im = make_float2(t.z, t.w);
                            tr[u] = fma2(both(ev.x), re, mul2(both(-ev.y), im));
                            ti[u] = fma2(both(ev.x), im, mul2(both(ev.y), re));
                        }
                    }
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        const float4 t = cp4[D == 3 ? N1 / 2 + v : v];
                        const float2 re = make_float2(t.x, t.y), im = make_float2(t.z, t.w);
#pragma unroll
                        for (int u = 0; u < NU; ++u) {
                            float ur = ev.x, ui = ev.y;
                            if constexpr (D == 3) {
                                ur = u & 1 ? tr[u / 2].y : tr[u / 2].x;
                                ui = u & 1 ? ti[u / 2].y : ti[u / 2].x;
                            }
                            accr[u][v] = fma2(both(ur), re, fma2(both(-ui), im, accr[u][v]));
                            acci[u][v] = fma2(both(ur), im, fma2(both(ui), re, acci[u][v]));
                        }
                    }
                }
#pragma unroll
                for (int u = 0; u < NU; ++u)
#pragma unroll
                    for (int v = 0; v < 2 * NV; ++v) {
                        const int r = D == 3 ? (kp * NA + u) * NK1 + v : v;
                        const float2 ar = accr[u][v / 2], ai = acci[u][v / 2];
                        if ((rows_in >> r) & 1ull)
                            atomicAdd(Wc + rowoff[r], v & 1 ? make_float2(ar.y, ai.y) : make_float2(ar.x, ai.x));
                    }
            }
        }
        if (tid == 0) fetched();
    }
}

// Exclusive scan of (binned packets, items) per key: a bin with at least
// kBinMinCount packets counts its packets and ceil(n / kBinT) items, other bins
// count zero.  off[K] receives the totals.
__device__ __forceinline__ int2 bin_pair(const int *count, int64_t k, int64_t K) {
    if (k >= K) return make_int2(0, 0);
    const int n = count[k];
    return n >= kBinMinCount ? make_int2(n, (n + kBinT - 1) / kBinT) : make_int2(0, 0);
}

__device__ __forceinline__ int2 block_exclusive_scan(int2 v, int2 *total) {
    __shared__ int2 wsum[32];  // (blockDim.x a multiple of 32, at most 1024)
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int2 x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int yx = __shfl_up_sync(0xffffffffu, x.x, o), yy = __shfl_up_sync(0xffffffffu, x.y, o);
        if (lane >= o) {
            x.x += yx;
            x.y += yy;
        }
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int2 w = lane < nw ? wsum[lane] : make_int2(0, 0);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int yx = __shfl_up_sync(0xffffffffu, w.x, o), yy = __shfl_up_sync(0xffffffffu, w.y, o);
            if (lane >= o) {
                w.x += yx;
                w.y += yy;
            }
        }
        if (lane < nw) wsum[lane] = w;  // inclusive warp prefixes
    }
    __syncthreads();
    const int2 before = wid > 0 ? wsum[wid - 1] : make_int2(0, 0);
    *total = wsum[nw - 1];
    __syncthreads();
    return make_int2(before.x + x.x - v.x, before.y + x.y - v.y);
}

__global__ void __launch_bounds__(1024) bin_scan1_kernel(const int *__restrict__ count, int64_t K,
                                                         int2 *__restrict__ off, int2 *__restrict__ bsum) {
    const int64_t k = blockIdx.x * (int64_t)1024 + threadIdx.x;
    int2 tot;
    const int2 e = block_exclusive_scan(bin_pair(count, k, K), &tot);
    if (k < K) off[k] = e;
    if (threadIdx.x == 0) bsum[blockIdx.x] = tot;
}

// One CTA: exclusive scan of the block totals (in place); off[K] = total.
__global__ void __launch_bounds__(1024) bin_scan2_kernel(int2 *__restrict__ bsum, int64_t nblk,
                                                         int2 *__restrict__ off, int64_t K) {
    int2 carry = make_int2(0, 0);
    for (int64_t b0 = 0; b0 < nblk; b0 += 1024) {
        const int64_t b = b0 + threadIdx.x;
        const int2 v = b < nblk ? bsum[b] : make_int2(0, 0);
        int2 tot;
        const int2 e = block_exclusive_scan(v, &tot);
        if (b < nblk) bsum[b] = make_int2(carry.x + e.x, carry.y + e.y);
        carry.x += tot.x;
        carry.y += tot.y;
    }
    if (threadIdx.x == 0) off[K] = carry;
}

__global__ void __launch_bounds__(1024) bin_scan3_kernel(int2 *__restrict__ off, int64_t K,
                                                         const int2 *__restrict__ bsum) {
    const int64_t k = blockIdx.x * (int64_t)1024 + threadIdx.x;
    if (k >= K) return;
    const int2 b = bsum[blockIdx.x];
    int2 v = off[k];
    v.x += b.x;
    v.y += b.y;
    off[k] = v;
}

// The binned scatter (FP32): binning, records and items, then the binned kernel
// and the per-packet kernel over the loose list, all on stream st.
template <int D, int N1>
fgr_status launch_binned_d(const BinLaunch &L, cudaStream_t st, const PacketsDev &pk, const Params32 &P, void *W,
                           uint8_t *flags, StageMarks *marks) {
    const int64_t m = pk.m, K = L.box.K;
    const BinBuffers &b = L.buf;
    FGR_CUDA_TRY(cudaMemsetAsync(b.count, 0, sizeof(int) * (size_t)K, st));
    FGR_CUDA_TRY(cudaMemsetAsync(b.ctr, 0, sizeof(int) * 4, st));
    if (D == 3) FGR_CUDA_TRY(cudaMemsetAsync(b.kbox, 0x7f, sizeof(int4) * (size_t)K, st));
    const unsigned pblocks = (unsigned)((m + 255) / 256), kblocks = (unsigned)((K + 255) / 256);
    bin_key_kernel<D><<<pblocks, 256, 0, st>>>(pk.q, pk.p, pk.a, m, P.c, L.box, b.key, b.rank, b.count);
    const int64_t nblk = (K + 1023) / 1024;
    bin_scan1_kernel<<<(unsigned)nblk, 1024, 0, st>>>(b.count, K, b.off, b.bsum);
    bin_scan2_kernel<<<1, 1024, 0, st>>>(b.bsum, nblk, b.off, K);
    bin_scan3_kernel<<<(unsigned)nblk, 1024, 0, st>>>(b.off, K, b.bsum);
    bin_place_kernel<D><<<pblocks, 256, 0, st>>>(pk.q, pk.p, pk.s, pk.a, m, P.c, L.split, b.key, b.rank, b.off, b.rec,
                                                 b.kbox, b.loose, b.ctr);
    // the rows and their boxes, and the clearing of those rows
    if (D == 3)
        FGR_CUDA_TRY(cudaMemsetAsync(L.row_box, 0x7f, sizeof(int4) * (size_t)L.rows, st));
    else
        FGR_CUDA_TRY(cudaMemsetAsync(L.row_range, 0x7f, sizeof(int2) * (size_t)L.rows * L.halves, st));
    const int per = K < (1 << 18) ? 8 : 1;
    bin_mark_rows_kernel<D><<<(unsigned)((K * per + 255) / 256), 256, 0, st>>>(b.count, b.kbox, P.c, L.box, per, flags,
                                                                             L.row_box, L.row_range, L.halves);
    // about 64 warps per SM: few long rows (d = 2: 5,796 of 37 KB) are cut into
    // parts (139 us with one warp per 32 rows, 19 us so), many short ones not
    const int64_t warps = (L.rows + 31) / 32, row_f4 = L.row_cells / 2;
    const int64_t parts = std::max<int64_t>(1, std::min<int64_t>((int64_t)L.num_sms * 64 / warps, (row_f4 + 31) / 32));
    const dim3 cgrid((unsigned)std::min<int64_t>((warps + 7) / 8, (int64_t)L.num_sms * 8),
                     (unsigned)std::min<int64_t>(parts, 65535));
    clear_flagged_rows_kernel<<<cgrid, 256, 0, st>>>((float4 *)W, flags, L.rows, row_f4);
    bin_items_kernel<D><<<kblocks, 256, 0, st>>>(b.off, b.kbox, P.c, L.box, b.items);
    FGR_CUDA_TRY(cudaGetLastError());
    if (marks) marks->binned();
    constexpr int smem = binned_smem_bytes<D, N1>();
    FGR_CUDA_TRY(cudaFuncSetAttribute(binned_scatter_kernel<D, N1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      smem));
    binned_scatter_kernel<D, N1><<<(unsigned)(L.num_sms * bin_ctas_per_sm<D>()), kBinT, smem, st>>>(
        P, L.box, b.rec, b.items, b.off + K, b.ctr + 1, (float2 *)W);
    constexpr int T = coeff_threads<false, N1>();
    coeff_scatter_list_kernel<D, false, N1><<<(unsigned)(L.num_sms * 4), T, 0, st>>>(
        pk.q, pk.p, pk.s, pk.a, m, P, W, flags, b.loose, b.ctr);
    FGR_CUDA_TRY(cudaGetLastError());
    return FGR_OK;
}

}  // namespace
}  // namespace fgr
