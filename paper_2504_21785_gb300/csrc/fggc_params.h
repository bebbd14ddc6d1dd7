// Parameter blocks of the FGGC kernels, shared by the node-box / grid-pass
// code (fggc.cu) and the coefficient + scatter kernels (fggc_coeff*.cu).
#pragma once

#include <algorithm>

#include "internal.h"

namespace fgr {

struct Common {
    int n1;
    int dq[kMaxN1], dp[kMaxN1];      // shifts, in orbit order (Lsa::order)
    int u3, v3;                      // orbits with |u|, |v| = 3/2 (Lsa::u3, v3)
    double dqv, dpv;                 // mesh steps
    double inv_dq, inv_dp;
    double cq2_4, cp2_4, cqcp_4;     // eq. 3.23 constants
    double cc;                       // cq cp / (2 pi): node phase in turns
    double inv_2pi_eps, pref;
    int amin[kMaxDim], A[kMaxDim], bmin[kMaxDim], B[kMaxDim];
    int64_t sa[kMaxDim], sb[kMaxDim];  // W strides of a_l and b_l
    int64_t row_len;                   // cells per row of the first grid pass
    int64_t ra[kMaxDim], rb[kMaxDim];  // sa / row_len, sb / row_len (dimensions before the last)
};

// Eigen factors of the least-squares problem (Lsa::sec, sec_inv, sec_one, kap_r, kap_i).
struct Factors64 {
    double sec[2][kMaxHalf * kMaxHalf], inv[2][kMaxHalf], one[kMaxHalf], kap_r[kMaxN1 / 4], kap_i[kMaxN1 / 4];
    int near;  // every Gaussian exponent of the right-hand side lies in [-1/4, 0], every half phase in [-3/32, 3/32]
};

inline Factors64 factors64(const Lsa &L) {
    Factors64 f;
    const double q = 0.5 * L.cq * (L.u3 ? 2.0 : 1.0), p = 0.5 * L.cp * (L.v3 ? 2.0 : 1.0);
    f.near = std::max(q, p) <= 0.5;
    for (int s = 0; s < 2; ++s) {
        for (int i = 0; i < kMaxHalf * kMaxHalf; ++i) f.sec[s][i] = L.sec[s][i];
        for (int i = 0; i < kMaxHalf; ++i) f.inv[s][i] = L.sec_inv[s][i];
    }
    for (int i = 0; i < kMaxHalf; ++i) f.one[i] = L.sec_one[i];
    for (int o = 0; o < kMaxN1 / 4; ++o) {
        f.kap_r[o] = L.kap_r[o];
        f.kap_i[o] = L.kap_i[o];
    }
    return f;
}

struct Params64 {
    Common c;
    Factors64 f;
};

struct Params32 {
    Common c;
    float poly[kSurTable];  // coefficient surrogate (Lsa::poly)
};

// Node box of one FGGC reconstruction and the sizes of its buffers.
struct FggcBox {
    Common c;               // constants and box (amin, A, bmin, B, strides)
    int64_t cells = 0;      // node cells
    int64_t rows0 = 0;      // rows of the first grid pass
    int64_t maxbuf = 0;     // elements of each pass buffer (d > 1)
    int64_t max_lines = 0;  // 8-byte entries of the b-ranges ((row, a) lines) or row boxes (two each)
    int64_t table_entries = 0;  // 8-byte entries of the pass tables of all dimensions
    int64_t fft_elems = 0;      // complex elements of the DFT lines of the largest pass (0: no DFT stage)
    bool empty = true;      // no packet reaches the grid
    bool apart = true;      // neighbouring packets mostly lie in cells more than two apart (d = 2)
};

struct FggcBuffers {
    void *W = nullptr, *buf1 = nullptr, *buf2 = nullptr;
    uint8_t *flags = nullptr;
    int2 *brange = nullptr;  // b-range per (row, a) line, or row boxes (int4) and ranges
    void *tables = nullptr;  // per-pass tables (node windows, point phases, tile bands)
    void *bin = nullptr;     // binning buffers of the FP32 scatter, d >= 2 (NULL: per-packet scatter)
    size_t bin_bytes = 0;    // bytes of the binning buffers
    unsigned long long *terms = nullptr;  // node-point terms of the passes (timed calls only)
    int2 *term_lines = nullptr;  // b-range per line for counting them (d >= 2)
    void *fft = nullptr;      // DFT lines of the commensurate grid stage (box.fft_elems complex)
    void *twiddle = nullptr;  // e^{2 pi i j / N}, j < N / 2 <= 4096 (complex)
};

// Binning of the FP32 scatter (fggc_bin.cuh).  A packet's key is the row-major
// index over its outer anchor (a0, b0) of dimensions 0..d-2, restricted to the
// anchors whose neighbours can reach the node box, and the kBinTileA x kBinTileB
// tile of its inner anchor (dimension d-1; d = 3: one tile).
struct BinBox {
    int ka_lo[3] = {}, KA[3] = {1, 1, 1}, kb_lo[3] = {}, KB[3] = {1, 1, 1};  // anchors per dimension
    int tiles_a = 1, tiles_b = 1;
    int dqmin = 0, dqmax = 0, dpmin = 0, dpmax = 0;  // neighbour shift ranges
    int64_t K = 0;                                   // keys
    bool boxes = false;                              // every key keeps its inner anchors' box (d = 3)
};

// Constants of a packet's record as unevaluated FP32 sums (see split_double).
struct SplitConst {
    float inv_dq[2], inv_dp[2], cc[2], half_cc[2], inv_2pi_eps[2], pref[2];
};

// A binned packet: per dimension the offsets (sx, ty) from its cell centre, the
// weight with the neighbour-independent phase, e^{i cq cp A / 2} of the inner
// dimension and the inner anchor relative to the node box.
struct BinRecord {
    float4 x;  // sx, ty of dimension 0, then of the last
    float4 w;  // weight, z of the last dimension
    float4 y;  // inner anchor (two ints), then sx, ty of dimension 1 (d = 3)
};

// Up to kBinT packets of one key: first record, packets, the inner target box
// [ta0, ta1] x [tb0, tb1] in the node box, and z of the outer dimensions.
struct BinItem {
    int4 at;   // key, first record, packets, 0
    int4 box;  // ta0, ta1, tb0, tb1
    float4 z;  // dimension 0, dimension 1
};

// Device buffers of the binning (m packets, K keys).
struct BinBuffers {
    int *key = nullptr;     // [m] key of each packet (-1: adds nothing)
    int *rank = nullptr;    // [m] place of the packet within its key
    int *loose = nullptr;   // [m] packets of small cells
    BinRecord *rec = nullptr;  // [m] records of the binned packets, by key
    int *count = nullptr;   // [K] packets per key
    int4 *kbox = nullptr;   // [K] min a, min -a, min b, min -b of the inner anchors per key (d = 3)
    int2 *off = nullptr;    // [K + 1] (first record, first item) per key; totals at K
    int2 *bsum = nullptr;   // [ceil(K / 1024)] block totals of the scan
    BinItem *items = nullptr;  // [max items]
    int *ctr = nullptr;     // [4] loose count, work counter
};

// b values per range of a row's nodes (fggc_rows.cuh).
constexpr int kRowHalf = 4;

struct BinLaunch {
    BinBox box;
    BinBuffers buf;
    SplitConst split;
    int num_sms = 1;
    // rows of W (each row_cells cells): only the rows that binned packets reach
    // are marked and zeroed
    int64_t rows = 0;
    int64_t row_cells = 0;
    // receive the inner nodes of every row: d = 3 its box, d = 2 the range of a per four b
    // values (halves of them), as grid_rows_kernel reads them
    int4 *row_box = nullptr;    // [rows]
    int2 *row_range = nullptr;  // [rows][halves]
    int halves = 0;
};

// Largest key box of the binned scatter; larger boxes use the per-packet kernel.
constexpr int64_t kMaxBinKeys = int64_t(1) << 26;
// Smallest bin (packets); smaller ones take the per-packet kernel.
constexpr int kBinMinCount = 8;
// d = 2: inner anchors per tile.  Larger tiles repeat fewer target cells at their
// edges, smaller ones give items that one CTA takes whole; at the flow's density
// of one packet per cell 24 x 16, 20 x 12 and 32 x 16 measured the same (2-D
// workload 1.37 ms), 16 x 12 1.43, 12 x 12 1.48 and 8 x 8 1.77 ms.
constexpr int kBinTileA = 24, kBinTileB = 16;
// Where the binned scatter runs in 2-D (whole calls, binned / per packet, in us).  The
// per-packet kernel's reductions meet in L2 where packets that follow each other lie in
// cells next to each other (mesh order), so the rule depends on the order, which the bounds
// kernel samples (order_probe).
// Apart: from kBinMinPackets2d (147,456 packets: n1 = 8 198 / 317, n1 = 4 185 / 197; 1.0M: 394
// / 1909 and 324 / 925), where the mean bin holds kBinMinMean2d packets (2.2: 656 / 448; 2.9:
// 536 / 434; 4.3: 758 / 740; 5.8: 604 / 664), half of that where the node array is beyond L2
// (kBinL2Cells; 2.0: 1086 / 1350).
// Near, n1 = 8: from kBinMinNear8 (147,456: 183 / 150; 262,144: 300 / 279 and 221 / 192; 419,904:
// 307 / 304; 1.6M: 590 / 762), mean kBinMinMeanNear.
// Near, n1 = 4: from kBinMinNear4 (1.0M: 380 / 330) where bins hold kBinMinFull packets (not
// scaled; 4.2M on 1024^2 points, 35 per bin: 1079 / 960; 54: 859 / 815; 178: 729 / 805; 17M,
// 173: 2319 / 3099), a third of that where the mean is kBinDense (1.0M: 191 / 291).
// The mean bin is scaled by the part of a tile that the inner plane fills: an item costs a
// CTA the same however few packets it holds, and on small planes the reductions are cheap
// (5 x 6 cells, 4.2M packets, 8 per bin: 4.6 / 3.2 ms; 24 per bin: 740 / 685 us; 48: 910 /
// 1196).
constexpr int64_t kBinMinPackets2d = 1 << 17, kBinMinNear8 = 1 << 18, kBinMinNear4 = 3 << 19;
constexpr int64_t kBinL2Cells = 1 << 24;
constexpr double kBinMinMean2d = 4.0, kBinMinMeanNear = 8.0, kBinMinFull = 96.0, kBinDense = 512.0;

// Key box of a node box and m packets (false when the binned scatter does not apply).
bool make_bin_box(const FggcBox &box, int d, int64_t m, BinBox *bb);
// Bytes of the binning buffers for m packets and key box bb.
size_t bin_buffer_bytes(int64_t m, const BinBox &bb);
// Carves the binning buffers out of one device block of bin_buffer_bytes.
void bin_buffers_at(void *block, int64_t m, const BinBox &bb, BinBuffers *out);

// Stage marks of the timed FGGC call (the binning ends where binned() is called).
struct StageMarks {
    StageTimer *timer = nullptr;
    double *slot = nullptr;
    void binned() {
        if (timer) timer->mark(slot);
    }
};

// Batched FGGC (fgr_reconstruct_fggc_batch): per-request parameters of one
// launch over up to kBatchMax requests of one dimension; CTA b of the launch
// belongs to the request r with block0[r] <= b < block0[r + 1].
constexpr int kBatchMax = 32;

struct ScatterBatchBase {
    int n;
    int block0[kBatchMax + 1];
    Common c[kBatchMax];
    const double *q[kBatchMax], *p[kBatchMax], *s[kBatchMax], *a[kBatchMax];
    int64_t m[kBatchMax];
    void *W[kBatchMax];
    uint8_t *flags[kBatchMax];
};
struct ScatterBatch64 : ScatterBatchBase {
    Factors64 f;
};
struct ScatterBatch32 : ScatterBatchBase {
    float poly[kSurTable];
};

// One request of a batched FGGC call: its context, planned box and buffers,
// bounds and overflow flag (device), packets and output (device).
struct FggcRequest {
    const fgr_ctx *ctx;
    const FggcBox *box;
    const FggcBuffers *buf;
    int *bnd, *overflow;
    PacketsDev pk;
    void *u;
};
// Enqueues the requests (any dimensions, one precision and neighbour
// strategy): per dimension and kBatchMax requests, one launch per stage.
fgr_status run_fggc_batch(int n, const FggcRequest *req, cudaStream_t st);

// Launches the batched per-packet coefficient + scatter kernel of dimension d
// (grid: batch.block0[batch.n] CTAs of coeff_threads); exactly one batch is non-NULL.
fgr_status launch_scatter_batch(int d, int n1, cudaStream_t st, const ScatterBatch64 *b64, const ScatterBatch32 *b32);
fgr_status launch_scatter_batch_d1(int n1, cudaStream_t st, const ScatterBatch64 *b64, const ScatterBatch32 *b32);
fgr_status launch_scatter_batch_d2(int n1, cudaStream_t st, const ScatterBatch64 *b64, const ScatterBatch32 *b32);
fgr_status launch_scatter_batch_d3(int n1, cudaStream_t st, const ScatterBatch64 *b64, const ScatterBatch32 *b32);
// Threads per CTA of the per-packet scatter kernel.
int scatter_threads(bool fp64, int n1);

// Box from the packets' node bounds hb[12] (per dimension: a min, a max, b min,
// b max), widened by margin nodes on every side, and their order hb[13] (of hb[14]).
fgr_status make_box(const fgr_ctx *ctx, const int *hb, int margin, FggcBox *box);

// Node bounds and order of the packets into hb[14] on the host (waits for them);
// bnd_dev: 14 device ints.
fgr_status compute_node_bounds(fgr_ctx *ctx, const PacketsDev &pk, int *bnd_dev, int *hb, cudaStream_t st);

// FGGC into u_dev with a planned box and buffers: stream-ordered only; sets
// *overflow (device) when the packets' nodes leave the box (their
// contributions outside it are then missing).  bnd: 12 device ints.
fgr_status run_fggc_planned(fgr_ctx *ctx, const PacketsDev &pk, const FggcBox &box, const FggcBuffers &b,
                            int *bnd, int *overflow, void *u_dev, cudaStream_t st);

// Launches the coefficient + scatter kernel (K3+K4) for dimension d, one
// thread per packet; exactly one of p64 / p32 is non-NULL.
fgr_status launch_coeff_scatter(int d, int n1, cudaStream_t st, const PacketsDev &pk, const Params64 *p64,
                                const Params32 *p32, void *W, uint8_t *flags);
fgr_status launch_coeff_scatter_d1(int n1, cudaStream_t st, const PacketsDev &pk, const Params64 *p64,
                                   const Params32 *p32, void *W, uint8_t *flags);
fgr_status launch_coeff_scatter_d2(int n1, cudaStream_t st, const PacketsDev &pk, const Params64 *p64,
                                   const Params32 *p32, void *W, uint8_t *flags);
fgr_status launch_coeff_scatter_d3(int n1, cudaStream_t st, const PacketsDev &pk, const Params64 *p64,
                                   const Params32 *p32, void *W, uint8_t *flags);
// The binned scatter (FP32, d = 2 or 3, n1 = 4 or 8): binning kernels, then the
// binned kernel and the per-packet kernel over the loose list.
fgr_status launch_binned_scatter(int d, int n1, const BinLaunch &L, cudaStream_t st, const PacketsDev &pk,
                                 const Params32 &P, void *W, uint8_t *flags, StageMarks *marks);
fgr_status launch_binned_d2(int n1, const BinLaunch &L, cudaStream_t st, const PacketsDev &pk, const Params32 &P,
                            void *W, uint8_t *flags, StageMarks *marks);
fgr_status launch_binned_d3(int n1, const BinLaunch &L, cudaStream_t st, const PacketsDev &pk, const Params32 &P,
                            void *W, uint8_t *flags, StageMarks *marks);

}  // namespace fgr
