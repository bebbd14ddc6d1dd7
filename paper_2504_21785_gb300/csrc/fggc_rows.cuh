// K5 for d >= 2 (FP32): one separable pass of eq. 2.24, rows [a][b] -> [m],
// with the output written in the layout the next pass reads.
//
// Every row knows which nodes it has: in the first pass the box (a-range x
// b-range) of its non-zero nodes, from the bins of the scatter (or a scan of W); in
// the next ones, per four b values, the range of a, from the rows that feed them
// and the node windows, for every kBoxPts points already contracted
// (row_range_kernel; position and momentum are correlated, so that the box of a
// row would be several times larger).  A pass reads and multiplies only those
// nodes, and writes only what the next pass reads, so the dead part of the node
// array (3 rows of 4 on the 3-D workload) is neither read nor written.
//
// A CTA takes kRowPts consecutive points and up to rpc rows that are consecutive
// b values of the next pass's lines.  The Gaussian factors g(x_m - a dq) of the
// tile's node band are tabulated once in shared memory.  A warp takes one row at
// a time, two points per lane: tiles of kRowB b values x 32 nodes arrive by
// cp.async.bulk.tensor (double-buffered per warp); per node the lane multiplies
// its two factors with kRowB complex values (two 16-byte broadcast loads per four
// values, one two-wide multiply-add per value and point) into kRowB x 2 sums.
// The sums over b follow by Horner's rule in e^{i dp x_m / eps} from the middle b
// of the tile, whose phase is reduced per point.  The CTA's results go through
// shared memory and leave transposed, rpc values in a piece.
//
// Bound by instruction issue: per node and four values 2 shared loads and 8
// two-wide multiply-adds.  Against one point per lane, whole 8 x 32 tiles over
// the band of a 32-point tile, a b-range scan before and a transpose after every
// pass: 3-D workload (16.8M packets, 256^3 points) grid stage 4.92 -> 2.42 ms,
// 2-D (4.2M, 1024^2) 0.54 -> 0.44 ms.
//
// Included by fggc.cu inside its anonymous namespace, after fggc_tma.cuh.
#pragma once

constexpr int kRowPts = 64;     // points per tile (two per lane)
constexpr int kBoxLog = 3;
constexpr int kBoxPts = 1 << kBoxLog;  // contracted points that share their ranges
constexpr int kRowB = 8;        // b values per tile
constexpr int kRowHalf = kRowB / 2;  // b values per range
constexpr int kRowLines = 32;   // nodes per tile
constexpr int kRowWarps = 4;
constexpr int kRowMax = 24;     // rows per CTA, at most
constexpr int kRowStage = kRowPts + 2;  // staged row, in float2 (16-byte rows)
constexpr size_t kRowSmemMax = 96 * 1024;

// Boxes and ranges hold minima: (min a, min -a, min b, min -b) and (min a, min -a);
// kBoxEmpty where there is nothing.
constexpr int kBoxEmpty = 0x7f7f7f7f;

struct RowPass {
    PassParams pp;
    // rows in groups of gl (consecutive b of a line of the next pass), parts CTAs per group
    int gl, parts, rpc;
    int lines;   // node lines of the factor table: at most min(band, A)
    int chunks;  // tiles of kRowB values in B
    const float2 *near;  // [N] offset from the nearest node, and its index
    // first pass: box[row]; else ranges[r * halves + b / kRowHalf], halves = ceil(B / kRowHalf),
    // of r = ((row / d1) >> s1) * stride + ((row % d1) >> s0)
    const int4 *box;
    const int2 *range;
    int64_t d1, stride;
    int s1, s0;
    // ranges of the next pass (null: the last pass, which writes everything): group o
    // feeds line o % next_lines of the rows with the ranges of
    // (point / kBoxPts) * next_groups + (o / next_lines >> next_shift)
    const int2 *next;
    int64_t next_groups;
    int next_lines, next_shift, next_halves;
};

inline size_t row_pass_smem(int lines, int rpc, int chunks) {
    return (size_t)kRowWarps * 2 * kRowLines * kRowB * sizeof(float2) + sizeof(float2) * (size_t)rpc * kRowStage +
           sizeof(int2) * (size_t)rpc * chunks + sizeof(float) * (size_t)lines * kRowPts;
}

// z <- z w + v (complex)
__device__ __forceinline__ void horner(float2 &z, float wr, float wi, float2 v) {
    const float re = fmaf(z.x, wr, fmaf(-z.y, wi, v.x));
    z.y = fmaf(z.x, wi, fmaf(z.y, wr, v.y));
    z.x = re;
}

__global__ void __launch_bounds__(kRowWarps * 32, 5) grid_rows_kernel(const __grid_constant__ CUtensorMap map,
                                                                      const __grid_constant__ CUtensorMap map_half,
                                                                      float2 *__restrict__ out,
                                                                      const __grid_constant__ RowPass R,
                                                                      const PassTables tab, int *__restrict__ err) {
    extern __shared__ __align__(128) unsigned char row_smem[];
    // tiles first: copies land on 128-byte boundaries
    float2(*sw)[2][kRowLines][kRowB] = reinterpret_cast<float2(*)[2][kRowLines][kRowB]>(row_smem);
    float2 *stage = reinterpret_cast<float2 *>(row_smem + (size_t)kRowWarps * 2 * kRowLines * kRowB * sizeof(float2));
    // per row and chunk of kRowB b values: first line (in the band) and lines, with
    // the halves that have any in the top bits of the first
    int2 *work = reinterpret_cast<int2 *>(stage + R.rpc * kRowStage);
    float *g = reinterpret_cast<float *>(work + R.rpc * R.chunks);
    __shared__ __align__(8) uint64_t bars[kRowWarps][2];
    const PassParams &pp = R.pp;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int tile = blockIdx.y;
    const int64_t o = blockIdx.x / R.parts;
    const int r0 = (int)(blockIdx.x % R.parts) * R.rpc, nr = min(R.rpc, R.gl - r0);
    if (R.next) {
        const int h0 = r0 / kRowHalf, nh = (r0 + nr - 1) / kRowHalf - h0 + 1, a = (int)(o % R.next_lines);
        const int64_t grp = o / R.next_lines >> R.next_shift;
        bool need = false;
        for (int e = tid; e < kRowPts / kBoxPts * nh; e += kRowWarps * 32) {
            const int s = tile * (kRowPts / kBoxPts) + e / nh, h = h0 + e % nh;
            if (s * kBoxPts >= pp.N) continue;
            const int2 *rg = R.next + (s * R.next_groups + grp) * R.next_halves;
            const int2 x = rg[h], y = (h ^ 1) < R.next_halves ? rg[h ^ 1] : make_int2(kBoxEmpty, kBoxEmpty);
            need = need || (x.x != kBoxEmpty && a >= min(x.x, y.x) && a <= -min(x.y, y.y));
        }
        if (!__syncthreads_or(need)) return;  // not read
    }
    const int64_t row0 = o * R.gl + r0;
    const int2 band = tab.band[tile];
    const int band0 = band.x - pp.amin;  // first node of the band
    bool any = false;
    for (int e = tid; e < nr * R.chunks; e += kRowWarps * 32) {
        const int r = e / R.chunks, k = e - r * R.chunks;
        const int64_t row = row0 + r;
        int lo = kBoxEmpty, hi = kBoxEmpty;  // min a, min -a
        unsigned halves = 0;
        if (R.box) {
            const int4 b = R.box[row];
            const int b0 = k * kRowB;
            if (b.x != kBoxEmpty && b.z < b0 + kRowB && -b.w >= b0) {
                lo = b.x;
                hi = b.y;
                halves = (b.z < b0 + kRowHalf ? 1u : 0u) | (-b.w >= b0 + kRowHalf ? 2u : 0u);
            }
        } else {
            const int64_t q = row / R.d1, m = row - q * R.d1;
            const int nh = (pp.B + kRowHalf - 1) / kRowHalf;
            const int2 *rg = R.range + ((q >> R.s1) * R.stride + (m >> R.s0)) * nh;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (2 * k + h < nh) {
                    const int2 x = rg[2 * k + h];
                    lo = min(lo, x.x);
                    hi = min(hi, x.y);
                    halves |= x.x != kBoxEmpty ? 1u << h : 0u;
                }
        }
        int l0 = 0, nl = 0;
        if (halves) {
            l0 = max(lo - band0, 0);
            nl = max(0, min(-hi, band.y - pp.amin) - band0 - l0 + 1);
        }
        work[e] = make_int2(l0 | (int)(halves << 30), nl);
        any = any || nl > 0;
    }
    any = __syncthreads_or(any);
    const int m = tile * kRowPts + 2 * lane;
    if (any) {
        // Gaussian factors of the band: thread = one point, every other line; dx from
        // the point's nearest node, so that it keeps FP32 relative accuracy
        {
            const int pt = tid % kRowPts, mp = tile * kRowPts + pt;
            const float2 nr2 = R.near[min((int64_t)mp, pp.N - 1)];
            const float dqf = (float)pp.dq;
            const float cef = (float)(pp.neg_half_inv_eps * 1.4426950408889634);  // log2(e) / (-2 eps)
            const int nb = min(R.lines, band.y - band.x + 1), off = band.x - __float_as_int(nr2.y);
            for (int j = tid / kRowPts; j < nb; j += kRowWarps * 32 / kRowPts) {
                const int2 w = tab.win[band0 + j];
                const float dx = fmaf((float)-(off + j), dqf, nr2.x);
                g[j * kRowPts + pt] = mp < pp.N && mp >= w.x && mp <= w.y ? ex2_approx(dx * dx * cef) : 0.f;
            }
        }
        if (lane == 0) {
            mbar_init(&bars[wid][0], 1);
            mbar_init(&bars[wid][1], 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fence_proxy_async_smem();
        }
    }
    __syncthreads();
    // per point: reduced phase of one b step, and its rotation w
    float2 ph[2];
    float wr[2], wi[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        ph[t] = tab.ph[min((int64_t)m + t, pp.N - 1)];
        sincospif(2.f * (ph[t].x - rint_fast(ph[t].x) + ph[t].y), &wi[t], &wr[t]);
    }
    // the warp's tiles: its rows, their chunks with lines, kRowLines lines at a time
    struct Cursor {
        int r, k, lc;
    };
    auto open = [&](Cursor &q, int2 &w) {  // the chunk at the cursor, or the next one with lines
        for (;; q.k = 0, q.r += kRowWarps) {
            if (q.r >= nr) return;
            for (; q.k < R.chunks; ++q.k) {
                w = work[q.r * R.chunks + q.k];
                if (w.y > 0) return;
            }
        }
    };
    int issued = 0, used = 0;
    Cursor ahead{wid, 0, 0};
    int2 aw = make_int2(0, 0);
    if (any) open(ahead, aw); else ahead.r = nr;
    auto issue = [&] {
        if (ahead.r >= nr) return;
        if (lane == 0) {
            const bool half = aw.y - ahead.lc <= kRowLines / 2;
            const int64_t line = (row0 + ahead.r) * (int64_t)pp.A + band0 + (aw.x & 0x3fffffff) + ahead.lc;
            uint64_t *bar = &bars[wid][issued & 1];
            mbar_expect_tx(bar, (half ? kRowLines / 2 : kRowLines) * kRowB * (int)sizeof(float2));
            tma_load_2d(&sw[wid][issued & 1][0][0], half ? &map_half : &map, ahead.k * kRowB, (int)line, bar);
        }
        ++issued;
        ahead.lc += kRowLines;
        if (ahead.lc >= aw.y) {
            ahead.lc = 0;
            ++ahead.k;
            open(ahead, aw);
        }
    };
    issue();
    issue();
    bool failed = false;
    for (int r = wid; r < nr; r += kRowWarps) {
        float2 sum[2] = {both(0.f), both(0.f)}, low[2] = {both(0.f), both(0.f)};  // Kahan sums
#pragma unroll 1
        for (int k = 0; k < R.chunks && any && !failed; ++k) {
            const int2 w = work[r * R.chunks + k];
            const int nl = w.y;
            if (nl == 0) continue;
            const unsigned halves = (unsigned)w.x >> 30;
            const int skip = halves == 2u ? kRowHalf : 0;  // only the second half
            const float *gl = g + (w.x & 0x3fffffff) * kRowPts + 2 * lane;
            float2 v[2][kRowB];
#pragma unroll
            for (int u = 0; u < kRowB; ++u) v[0][u] = v[1][u] = both(0.f);
#pragma unroll 1
            for (int lc = 0; lc < nl; lc += kRowLines) {
                const int s = used & 1;
                if (!tma_wait(&bars[wid][s], (unsigned)(used >> 1) & 1u, err)) {
                    failed = true;
                    break;
                }
                ++used;
                const int n = min(kRowLines, nl - lc);
                const float *gj = gl + lc * kRowPts;
                const float4 *wj = reinterpret_cast<const float4 *>(&sw[wid][s][0][skip]);
                auto line = [&](auto nb) {
                    const float2 gg = *reinterpret_cast<const float2 *>(gj);
#pragma unroll
                    for (int u = 0; u < decltype(nb)::value / 2; ++u) {
                        const float4 x = wj[u];
                        const float2 w0 = make_float2(x.x, x.y), w1 = make_float2(x.z, x.w);
                        v[0][2 * u] = fma2(both(gg.x), w0, v[0][2 * u]);
                        v[1][2 * u] = fma2(both(gg.y), w0, v[1][2 * u]);
                        v[0][2 * u + 1] = fma2(both(gg.x), w1, v[0][2 * u + 1]);
                        v[1][2 * u + 1] = fma2(both(gg.y), w1, v[1][2 * u + 1]);
                    }
                    gj += kRowPts;
                    wj += kRowB / 2;
                };
                if (halves == 3u) {
#pragma unroll 2
                    for (int j = 0; j < n; ++j) line(std::integral_constant<int, kRowB>());
                } else {
#pragma unroll 2
                    for (int j = 0; j < n; ++j) line(std::integral_constant<int, kRowHalf>());
                }
                // the buffer is free again
                __syncwarp();
                if (lane == 0) fence_proxy_async_smem();
                issue();
            }
            if (failed) break;
            const float bf = (float)(pp.bmin + k * kRowB + skip + 3);
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                float2 z = v[t][0];
                horner(z, wr[t], -wi[t], v[t][1]);
                horner(z, wr[t], -wi[t], v[t][2]);
                horner(z, wr[t], -wi[t], v[t][3]);
                if (halves == 3u) {
                    float2 f = v[t][7];
                    horner(f, wr[t], wi[t], v[t][6]);
                    horner(f, wr[t], wi[t], v[t][5]);
                    horner(f, wr[t], wi[t], v[t][4]);
                    horner(f, wr[t], wi[t], z);
                    z = f;
                }
                float e = bf * ph[t].x;
                e -= rint_fast(e);
                float tau = fmaf(bf, ph[t].y, e);
                tau -= rint_fast(tau);
                float er, ei;
                sincospif(2.f * tau, &ei, &er);  // (shared by 8 b values: the fast one's 4e-7 would show)
                kahan_add(sum[t].x, low[t].x, er * z.x - ei * z.y);
                kahan_add(sum[t].y, low[t].y, er * z.y + ei * z.x);
            }
        }
        *reinterpret_cast<float4 *>(stage + r * kRowStage + 2 * lane) =
            make_float4(__fsub_rn(sum[0].x, low[0].x), __fsub_rn(sum[0].y, low[0].y), __fsub_rn(sum[1].x, low[1].x),
                        __fsub_rn(sum[1].y, low[1].y));
    }
    if (failed)  // leave only after this warp's copies in flight have landed (bounded)
        for (; used < issued; ++used)
            if (!tma_wait(&bars[wid][used & 1], (unsigned)(used >> 1) & 1u, err)) break;
    __syncthreads();
    for (int e = tid; e < nr * kRowPts; e += kRowWarps * 32) {
        const int pt = e / nr, r = e - pt * nr;
        const int64_t mp = (int64_t)tile * kRowPts + pt;
        if (mp < pp.N) out[mp * pp.rows + row0 + r] = stage[r * kRowStage + pt];
    }
}

// Ranges of the rows of the next pass (see RowPass): of the members i of group
// g, (a, b) = (i / B, i % B) in the next pass's dimension, those whose nodes
// reach the points of tile t through their windows (win: first and last point of
// every node) widen out[(t * groups + g) * halves + b / kRowHalf] by a.  A
// member's nodes: box[g * members + i], or range[(g * members + i) * in_halves ...].
// Eight lanes per member share out its tiles.
__global__ void __launch_bounds__(128) row_range_kernel(const int4 *__restrict__ box, const int2 *__restrict__ range,
                                                        int in_halves, int members, int B, int64_t groups,
                                                        const int2 *__restrict__ win, int halves, int2 *out) {
    const int64_t g = blockIdx.x;
    const int i = blockIdx.y * (blockDim.x / 8) + threadIdx.x / 8;
    if (i >= members) return;
    int lo = kBoxEmpty, hi = kBoxEmpty;
    if (box) {
        const int4 b = box[g * members + i];
        lo = b.x;
        hi = b.y;
    } else {
        for (int h = 0; h < in_halves; ++h) {
            const int2 x = range[(g * members + i) * in_halves + h];
            lo = min(lo, x.x);
            hi = min(hi, x.y);
        }
    }
    if (lo == kBoxEmpty) return;
    const int first = max(0, win[lo].x), last = win[-hi].y;  // windows ascend with the node
    const int a = i / B, h = (i - a * B) / kRowHalf;
    for (int t = (first >> kBoxLog) + threadIdx.x % 8; t << kBoxLog <= last; t += 8) {
        int2 *x = out + (t * groups + g) * halves + h;
        const int2 now = __ldcg(x);  // (a stale read only costs an atomic)
        if (a < now.x) atomicMin(&x->x, a);
        if (-a < now.y) atomicMin(&x->y, -a);
    }
}

// Boxes of the rows of W by reading the flagged ones (the per-packet scatter):
// one warp per row.
__global__ void __launch_bounds__(256) row_scan_kernel(const float2 *__restrict__ W, int64_t rows, int A, int B,
                                                       const uint8_t *__restrict__ flags, int4 *__restrict__ box) {
    const int lane = threadIdx.x & 31;
    const int64_t row = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
    if (row >= rows) return;
    int4 v = make_int4(kBoxEmpty, kBoxEmpty, kBoxEmpty, kBoxEmpty);
    if (flags[row]) {
        const float2 *p = W + row * (int64_t)A * B;
        const int cells = A * B;
        for (int e = lane; e < cells; e += 32) {
            const float2 x = p[e];
            if (x.x != 0.f || x.y != 0.f) {
                const int a = e / B, b = e - a * B;
                v.x = min(v.x, a);
                v.y = min(v.y, -a);
                v.z = min(v.z, b);
                v.w = min(v.w, -b);
            }
        }
    }
    v.x = __reduce_min_sync(0xffffffffu, v.x);
    v.y = __reduce_min_sync(0xffffffffu, v.y);
    v.z = __reduce_min_sync(0xffffffffu, v.z);
    v.w = __reduce_min_sync(0xffffffffu, v.w);
    if (lane == 0) box[row] = v;
}
