// K5 for d >= 2: one separable pass of eq. 2.24, rows [a][b] -> [m],
// with the output written in the layout the next pass reads.
//
// Every row knows which nodes it has: per four b values the range of a (position and
// momentum are correlated, so that the box of a row would be several times larger).  In
// the first pass from a scan of W or, after the binned scatter, from the bins (d = 3: the
// row's box); in the next ones from the rows that feed them and the node windows, for
// every kBoxPts points already contracted (row_range_kernel).  A pass reads and multiplies only those
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
// FP64: one point per lane, and the phases (rotation of a step, and of the middle b
// of every four) from a table of the pass instead of a sine and cosine per b, point
// and row; the FP64 pipe binds (94 %): 2-D Q2P2 set of 705,600 packets on 301 x 257
// points 2.42 -> 0.84 ms for both passes (1.48 with up to 24 rows per CTA whatever the
// wave covers).
//
// FP32: bound by instruction issue: per node and four values 2 shared loads and 8
// two-wide multiply-adds.  Against one point per lane, whole 8 x 32 tiles over
// the band of a 32-point tile, a b-range scan before and a transpose after every
// pass: 3-D workload (16.8M packets, 256^3 points) grid stage 4.92 -> 2.50 ms,
// 2-D (4.2M, 1024^2) 0.54 -> 0.41 ms.
//
// Included by fggc.cu inside its anonymous namespace, after fggc_tma.cuh.
#pragma once

// points per lane and per tile
template <bool FP64>
__host__ __device__ constexpr int row_ppl() {
    return FP64 ? 1 : 2;
}
template <bool FP64>
__host__ __device__ constexpr int row_pts() {
    return 32 * row_ppl<FP64>();
}
constexpr int kBoxLog = 3;
constexpr int kBoxPts = 1 << kBoxLog;  // contracted points that share their ranges
constexpr int kRowB = 8;        // b values per tile
static_assert(kRowB == 2 * kRowHalf, "a tile holds two ranges");
constexpr int kRowLines = 32;   // nodes per tile
constexpr int kRowWarps = 4;
constexpr int kRowMax = 24;     // rows per CTA, at most
// staged row, in complex values (16-byte rows, off the bank period)
template <bool FP64>
__host__ __device__ constexpr int row_stage() {
    return row_pts<FP64>() + (FP64 ? 1 : 2);
}
constexpr size_t kRowSmemMax = 96 * 1024;
// Slices of a pass's b range: up to this many warps per SM, of at least this many chunks.
constexpr int kRowSliceWarps = 16, kRowSliceChunks = 4;

// Boxes and ranges hold minima: (min a, min -a, min b, min -b) and (min a, min -a);
// kBoxEmpty where there is nothing.
constexpr int kBoxEmpty = 0x7f7f7f7f;

struct RowPass {
    PassParams pp;
    // rows in groups of gl (consecutive b of a line of the next pass), parts CTAs per group
    int gl, parts, rpc;
    int per;     // chunks per slice (blockIdx.z), where slices share out a row's chunks
    int lines;   // node lines of the factor table: at most min(band, A)
    int chunks;  // tiles of kRowB values in B
    const float2 *near;   // FP32: [N] offset from the nearest node, and its index
    const double2 *phase;  // FP64: [N] rotation of one b step, then [halves][N] phases of the middle b's
    // ranges[r * halves + b / kRowHalf], halves = ceil(B / kRowHalf), of
    // r = ((row / d1) >> s1) * stride + ((row % d1) >> s0); or box[row]
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

template <bool FP64>
inline size_t row_pass_smem(int lines, int rpc, int chunks) {
    const size_t c2 = FP64 ? 16 : 8;
    return (size_t)kRowWarps * 2 * kRowLines * kRowB * c2 + c2 * (size_t)rpc * row_stage<FP64>() +
           sizeof(int2) * (size_t)rpc * chunks + c2 / 2 * (size_t)lines * row_pts<FP64>();
}

// z <- z w + v (complex)
template <class C2, class Real>
__device__ __forceinline__ void horner(C2 &z, Real wr, Real wi, C2 v) {
    const Real re = fma(z.x, wr, fma(-z.y, wi, v.x));
    z.y = fma(z.x, wi, fma(z.y, wr, v.y));
    z.x = re;
}

// SLICED: blockIdx.z takes R.per of the chunks and adds to the output (cleared before).
template <bool FP64, bool SLICED>
__global__ void __launch_bounds__(kRowWarps * 32, FP64 ? 4 : 5)
    grid_rows_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap map_half,
                     typename std::conditional<FP64, double2, float2>::type *__restrict__ out,
                     const __grid_constant__ RowPass R, const PassTables tab, int *__restrict__ err) {
    using Real = typename std::conditional<FP64, double, float>::type;
    using C2 = typename std::conditional<FP64, double2, float2>::type;
    constexpr int kRowPts = row_pts<FP64>(), kRowStage = row_stage<FP64>(), PPL = row_ppl<FP64>();
    extern __shared__ __align__(128) unsigned char row_smem[];
    // tiles first: copies land on 128-byte boundaries
    C2(*sw)[2][kRowLines][kRowB] = reinterpret_cast<C2(*)[2][kRowLines][kRowB]>(row_smem);
    C2 *stage = reinterpret_cast<C2 *>(row_smem + (size_t)kRowWarps * 2 * kRowLines * kRowB * sizeof(C2));
    // per row and chunk of kRowB b values: first line (in the band) and lines, with
    // the halves that have any in the top bits of the first
    int2 *work = reinterpret_cast<int2 *>(stage + R.rpc * kRowStage);
    Real *g = reinterpret_cast<Real *>(work + R.rpc * R.chunks);
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
    const int k_first = SLICED ? (int)blockIdx.z * R.per : 0, k_end = k_first + R.per;
    bool any = false;
    for (int e = tid; e < nr * R.chunks; e += kRowWarps * 32) {
        const int r = e / R.chunks, k = e - r * R.chunks;
        const int64_t row = row0 + r;
        int lo = kBoxEmpty, hi = kBoxEmpty;  // min a, min -a
        unsigned halves = 0;
        if (SLICED && (k < k_first || k >= k_end)) {
            // another slice's
        } else if (R.box) {
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
    if (SLICED && !any) return;
    const int m = tile * kRowPts + PPL * lane;
    if (any) {
        // Gaussian factors of the band: thread = one point, every other line; dx from
        // the point's nearest node, so that it keeps FP32 relative accuracy
        {
            const int pt = tid % kRowPts, mp = tile * kRowPts + pt;
            const int64_t mc = min((int64_t)mp, pp.N - 1);
            const int nb = min(R.lines, band.y - band.x + 1);
            const float2 near = FP64 ? make_float2(0.f, 0.f) : R.near[mc];
            const double xm = FP64 ? grid_x(pp.lo, pp.h, mc) : 0.0;
            const float dqf = (float)pp.dq;
            const float cef = (float)(pp.neg_half_inv_eps * 1.4426950408889634);  // log2(e) / (-2 eps)
            for (int j = tid / kRowPts; j < nb; j += kRowWarps * 32 / kRowPts) {
                const int2 w = tab.win[band0 + j];
                Real v = 0;
                if (mp < pp.N && mp >= w.x && mp <= w.y) {
                    if constexpr (FP64) {
                        const double dx = xm - (double)(band.x + j) * pp.dq;
                        v = exp(dx * dx * pp.neg_half_inv_eps);
                    } else {
                        const float dx = fmaf((float)(__float_as_int(near.y) - band.x - j), dqf, near.x);
                        v = ex2_approx(dx * dx * cef);
                    }
                }
                g[j * kRowPts + pt] = v;
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
    // per point: rotation w of one b step (FP32: and its reduced phase)
    float2 ph[PPL];
    Real wr[PPL], wi[PPL];
#pragma unroll
    for (int t = 0; t < PPL; ++t) {
        const int64_t mc = min((int64_t)m + t, pp.N - 1);
        if constexpr (FP64) {
            const double2 w = R.phase[mc];
            wr[t] = w.x;
            wi[t] = w.y;
        } else {
            ph[t] = tab.ph[mc];
            sincospif(2.f * (ph[t].x - rint_fast(ph[t].x) + ph[t].y), &wi[t], &wr[t]);
        }
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
            mbar_expect_tx(bar, (half ? kRowLines / 2 : kRowLines) * kRowB * (int)sizeof(C2));
            // (FP64: the map's elements are the parts)
            tma_load_2d(&sw[wid][issued & 1][0][0], half ? &map_half : &map, ahead.k * kRowB * (FP64 ? 2 : 1), (int)line,
                        bar);
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
        C2 zero;
        zero.x = zero.y = 0;
        C2 sum[PPL], low[PPL];  // (FP32: Kahan sums)
#pragma unroll
        for (int t = 0; t < PPL; ++t) sum[t] = low[t] = zero;
#pragma unroll 1
        for (int k = 0; k < R.chunks && any && !failed; ++k) {
            const int2 w = work[r * R.chunks + k];
            const int nl = w.y;
            if (nl == 0) continue;
            const unsigned halves = (unsigned)w.x >> 30;
            const int skip = halves == 2u ? kRowHalf : 0;  // only the second half
            const Real *gl = g + (w.x & 0x3fffffff) * kRowPts + PPL * lane;
            C2 v[PPL][kRowB];
#pragma unroll
            for (int t = 0; t < PPL; ++t)
#pragma unroll
                for (int u = 0; u < kRowB; ++u) v[t][u] = zero;
#pragma unroll 1
            for (int lc = 0; lc < nl; lc += kRowLines) {
                const int s = used & 1;
                if (!tma_wait(&bars[wid][s], (unsigned)(used >> 1) & 1u, err)) {
                    failed = true;
                    break;
                }
                ++used;
                const int n = min(kRowLines, nl - lc);
                const Real *gj = gl + lc * kRowPts;
                const C2 *wj = &sw[wid][s][0][skip];
                auto line = [&](auto nb) {
                    Real gg[PPL];
                    if constexpr (FP64) {
                        gg[0] = *gj;
                    } else {
                        const float2 x = *reinterpret_cast<const float2 *>(gj);
                        gg[0] = x.x;
                        gg[1] = x.y;
                    }
#pragma unroll
                    for (int u = 0; u < decltype(nb)::value; u += 2) {
                        C2 x[2];  // two values: 16-byte loads
                        if constexpr (FP64) {
                            x[0] = wj[u];
                            x[1] = wj[u + 1];
                        } else {
                            const float4 y = *reinterpret_cast<const float4 *>(wj + u);
                            x[0] = make_float2(y.x, y.y);
                            x[1] = make_float2(y.z, y.w);
                        }
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int t = 0; t < PPL; ++t) scaled_add(v[t][u + h], gg[t], x[h]);
                    }
                    gj += kRowPts;
                    wj += kRowB;
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
            for (int t = 0; t < PPL; ++t) {
                C2 z = v[t][0];
                horner(z, wr[t], -wi[t], v[t][1]);
                horner(z, wr[t], -wi[t], v[t][2]);
                horner(z, wr[t], -wi[t], v[t][3]);
                if (halves == 3u) {
                    C2 f = v[t][7];
                    horner(f, wr[t], wi[t], v[t][6]);
                    horner(f, wr[t], wi[t], v[t][5]);
                    horner(f, wr[t], wi[t], v[t][4]);
                    horner(f, wr[t], wi[t], z);
                    z = f;
                }
                if constexpr (FP64) {
                    const int64_t mc = min((int64_t)m + t, pp.N - 1);
                    const double2 e = R.phase[(1 + 2 * k + (skip ? 1 : 0)) * pp.N + mc];
                    sum[t].x = fma(e.x, z.x, fma(-e.y, z.y, sum[t].x));
                    sum[t].y = fma(e.x, z.y, fma(e.y, z.x, sum[t].y));
                } else {
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
        }
        if constexpr (FP64) {
            stage[r * kRowStage + lane] = sum[0];
        } else {
            *reinterpret_cast<float4 *>(stage + r * kRowStage + 2 * lane) =
                make_float4(__fsub_rn(sum[0].x, low[0].x), __fsub_rn(sum[0].y, low[0].y),
                            __fsub_rn(sum[1].x, low[1].x), __fsub_rn(sum[1].y, low[1].y));
        }
    }
    if (failed)  // leave only after this warp's copies in flight have landed (bounded)
        for (; used < issued; ++used)
            if (!tma_wait(&bars[wid][used & 1], (unsigned)(used >> 1) & 1u, err)) break;
    __syncthreads();
    for (int e = tid; e < nr * kRowPts; e += kRowWarps * 32) {
        const int pt = e / nr, r = e - pt * nr;
        const int64_t mp = (int64_t)tile * kRowPts + pt;
        if (mp >= pp.N) continue;
        C2 *to = out + (mp * pp.rows + row0 + r);
        const C2 v = stage[r * kRowStage + pt];
        if (SLICED)
            atomic_add_c(to, v.x, v.y);
        else
            *to = v;
    }
}

// Ranges of the rows of the next pass (see RowPass): of the members i of group
// g, (a, b) = (i / B, i % B) in the next pass's dimension, those whose nodes
// reach the points of tile t through their windows (win: first and last point of
// every node) widen out[(t * groups + g) * halves + b / kRowHalf] by a.  A
// member's nodes: box[g * members + i], or range[(g * members + i) * in_halves ...].
// 1 << log_lanes lanes per member share out its tiles (one where there is a single tile:
// 530,000 members 104 -> 35 us against eight); part p of a group has consecutive
// members.
__global__ void __launch_bounds__(128) row_range_kernel(const int4 *__restrict__ box, const int2 *__restrict__ range,
                                                        int in_halves, int members, int log_lanes, int B,
                                                        int64_t groups, const int2 *__restrict__ win, int halves,
                                                        int2 *out) {
    // (neighbouring CTAs of different groups, whose ranges are apart: 3-D workload 67 -> 28 us)
    const int64_t g = blockIdx.x % (unsigned)groups;
    const int i = (int)(((blockIdx.x / (unsigned)groups) * blockDim.x + threadIdx.x) >> log_lanes);
    const int lanes = 1 << log_lanes;
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
    for (int t = (first >> kBoxLog) + (int)(threadIdx.x & (lanes - 1)); t << kBoxLog <= last; t += lanes) {
        int2 *x = out + (t * groups + g) * halves + h;
        const int2 now = __ldcg(x);  // (a stale read only costs an atomic)
        if (a < now.x) atomicMin(&x->x, a);
        if (-a < now.y) atomicMin(&x->y, -a);
    }
}

// Ranges of a per row of W and four b values (see RowPass) by reading the flagged rows
// (the per-packet scatter): LANES lanes take as many consecutive b values of a row, line
// after line (few where B is small: 530,000 rows of 40 cells 126 -> 59 us), and
// blockIdx.y of gridDim.y a part of the lines: rows too few to fill the device are cut,
// and their ranges, empty before, take the parts' minima.
template <class C2, int LANES>
__global__ void __launch_bounds__(256) row_scan_kernel(const C2 *__restrict__ W, int64_t rows, int A, int B,
                                                       int chunks, int halves, const uint8_t *__restrict__ flags,
                                                       int2 *__restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)(256 / LANES) + threadIdx.x / LANES;
    const int64_t row = i / chunks;
    const int b = (int)(i - row * chunks) * LANES + threadIdx.x % LANES;
    int lo = kBoxEmpty, hi = kBoxEmpty;  // min a, min -a
    if (row < rows && b < B && flags[row]) {
        const int part = (A - 1) / (int)gridDim.y + 1, a0 = (int)blockIdx.y * part, a1 = min(A, a0 + part);
        const C2 *p = W + (row * A + a0) * (int64_t)B + b;
#pragma unroll 8
        for (int a = a0; a < a1; ++a, p += B) {
            const C2 x = *p;
            if (x.x != 0 || x.y != 0) {
                lo = min(lo, a);
                hi = -a;
            }
        }
    }
#pragma unroll
    for (int o = 1; o < kRowHalf; o *= 2) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = min(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (threadIdx.x % kRowHalf > 0 || row >= rows || b >= B) return;
    int2 *x = out + row * halves + b / kRowHalf;
    if (gridDim.y == 1) {
        *x = make_int2(lo, hi);
    } else if (lo != kBoxEmpty) {
        atomicMin(&x->x, lo);
        atomicMin(&x->y, hi);
    }
}
