// Internal declarations of libfgr (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <string>

#include "fgr.h"

namespace fgr {

constexpr int kMaxDim = 3;
constexpr int kMaxN1 = 16;  // 1-D neighbours per packet: nq * np <= 16
constexpr int kMaxHalf = kMaxN1 / 2;

// FP32 coefficient surrogate: Chebyshev degree per variable and total degree.
// The terms T_i T_j with i + j <= surrogate_total and i, j < kCheb are kept for
// n1 <= 8 (Q2P2, Q4P2, Q2P4); their dropped coefficients sum to 1.1e-8 (Q4P2)
// and 1.1e-11 (Q2P2) of the largest one, under the FP32 rounding of the
// evaluation (2e-8 rms measured); n1 = 16 (Q4P4) keeps every i, j < kCheb.
constexpr int kCheb = 10;
template <int N1>
__host__ __device__ constexpr int surrogate_total() {
    return N1 <= 8 ? 11 : 2 * (kCheb - 1);
}
// Even (or odd) powers per variable in one parity part of the surrogate.
constexpr int kPow = kCheb / 2;
// Floats of the surrogate of one orbit of four mirrored neighbours:
// [re, im][parity part ee, oe, eo, oo][power of X^2][power of Y^2].
constexpr int kOrbitTable = 2 * 4 * kPow * kPow;
constexpr int kSurTable = kMaxN1 / 4 * kOrbitTable;

// The eps-free least-squares problem of eq. 3.22-3.23 of one neighbour strategy.
// The pseudo-inverse of its Gram matrix is applied through eigen factors.
struct Lsa {
    int nq = 4, np = 2, n1 = 8, rank = 0;
    double cq = 0.5, cp = 0.0;
    int dq[kMaxN1] = {}, dp[kMaxN1] = {};  // shifts, k = iq*np + ip
    double lam[kMaxN1] = {};               // eigenvalues, descending
    // Eigen factors by sector (even, odd under parity) in the real basis of
    // build_lsa: sec[s][a * kMaxHalf + i] = component a of eigenvector i, and
    // 1 / (4 lambda_i) above the cut-off, else 0.
    double sec[2][kMaxHalf * kMaxHalf] = {}, sec_inv[2][kMaxHalf] = {};
    // The even eigenvectors' products with a right-hand side of ones (coeff_dim64).
    double sec_one[kMaxHalf] = {};
    // Per orbit: e^{i cq cp |u v| / 2}.
    double kap_r[kMaxN1 / 4] = {}, kap_i[kMaxN1 / 4] = {};
    // Neighbours in orbit order: orbit o holds, at 4 o + g, the mirror images
    // (u, v), (u, -v), (-u, v), (-u, -v) of one shift, (u, v) = (dq - 1/2, dp - 1/2)
    // with u, v < 0 for g = 0 (the kernels number their neighbours this way).
    int order[kMaxN1] = {};
    int u3 = 0, v3 = 0;  // bit o: orbit o has |u|, |v| = 3/2 (else 1/2)
    // Surrogate of the first neighbour of every orbit (see build_lsa).
    float poly[kSurTable] = {};
};

// Builds Lsa (host, long double Jacobi).  Returns false on bad input.
bool build_lsa(double cq, double cp, int nq, int np, double rcond, Lsa *out);

struct Grid {
    int d = 1;
    int64_t n[kMaxDim] = {1, 1, 1};
    double lo[kMaxDim] = {}, hi[kMaxDim] = {}, h[kMaxDim] = {};
    int64_t total = 1;
};

struct Mesh {
    double eps, sigma, dq, dp, cq, cp, cqcp, pref, R, rs;  // rs = R*sqrt(eps)
};

struct Timing {
    bool enabled = false;
    bool count_terms = false;  // also count the grid passes' node-point terms (a scan and a count per pass,
                               // after the last stage)
    fgr_stats last{};
};

// Launch-shape parameters picked by the autotuner (autotune.cu).
struct Tuning {
    int direct_ctas_per_sm = 8;  // direct sum: tiles x slices >= this x SMs
    int pass_ctas_per_sm = 16;   // grid passes: rows x tiles x b-slices >= this x SMs
    int pass_tile = 0;           // grid points per grid-pass CTA: 32, 128, or 0 (by the band width)
    // pass_tile was set by the caller (fgr_set_tuning): 128 then also keeps d >= 2 calls off
    // grid_rows_kernel; a tuned 128 only shapes the pass kernels where that one does not apply
    bool tile_fixed = false;
};

// Seeds a new context's tuning from the process-wide table (autotune.cu).
void seed_tuning(fgr_ctx *ctx);

}  // namespace fgr

struct fgr_ctx {
    int d = 1;
    int device = 0;
    int num_sms = 1;
    fgr::Grid grid;
    fgr::Mesh mesh;
    fgr::Lsa lsa;
    fgr_options opt{};
    cudaMemPool_t pool = nullptr;
    fgr::Timing timing;
    fgr::Tuning tune;
    int fft_logn[fgr::kMaxDim] = {0, 0, 0};  // log2 N of the DFT grid stage per dimension (0: direct stage)
    int *dev_err = nullptr;          // device word: a kernel's bounded wait gave up (reported by the next call)
    // Device view of a host word (set by the server around a large direct
    // sum): while it is > 0 the persistent direct-sum CTAs past one per SM
    // stop between work items, so that waiting small requests get SM slots.
    const volatile int *yield_flag = nullptr;
    // Bytes that a call may take for buffers it can do without (partial sums of the 1-D
    // direct sum, binning of the 2-D FGGC scatter): the server's requests have what was
    // reserved for them within the budget.
    size_t spare_bytes = SIZE_MAX;
    bool *rows_probe = nullptr;  // set by the autotuner: true when grid_rows_kernel served a call
    int64_t *host_pinned = nullptr;  // small pinned buffer for device->host sizes
};

namespace fgr {

// thread-local error message
void set_error(const char *fmt, ...);
void clear_error();

#define FGR_CUDA_TRY(expr)                                                              \
    do {                                                                                \
        cudaError_t err__ = (expr);                                                     \
        if (err__ != cudaSuccess) {                                                     \
            ::fgr::set_error("%s failed: %s (%s:%d)", #expr, cudaGetErrorString(err__), \
                             __FILE__, __LINE__);                                       \
            return FGR_E_CUDA;                                                          \
        }                                                                               \
    } while (0)

// Device view of a packet set (device pointers).
struct PacketsDev {
    int64_t m;
    const double *q, *p, *s, *a;
};

// Stream-ordered scratch from the context's pool, released when the guard dies.
class Scratch {
  public:
    Scratch(fgr_ctx *ctx, cudaStream_t s) : ctx_(ctx), s_(s) {}
    ~Scratch();
    // returns nullptr and sets the error on failure
    void *get(size_t bytes);

  private:
    fgr_ctx *ctx_;
    cudaStream_t s_;
    void *ptrs_[32] = {};
    int n_ = 0;
};

// Kernel-stage launchers (return FGR_OK or an error with the message set).
fgr_status run_propagate(fgr_ctx *ctx, double *q, double *p, double *s, double *a, int64_t m,
                         const fgr_potential *v, double t, double dt, cudaStream_t st);
// Eq. 2.6 / 2.8 on the grid: a (2 x m) and s (m) of the packets at (q, p) from
// the wave u_dev (complex, the context's precision).
fgr_status run_decompose(fgr_ctx *ctx, const void *u_dev, const double *q, const double *p, double *s, double *a,
                         int64_t m, cudaStream_t st);
// One dimension of a tensor-product mesh (device pointers).
struct AxisDev {
    int64_t L;
    const double *q, *p;
};
// Eq. 2.8 onto the tensor product of d lists: a (2 x m) of the packets with
// row-major indices sel[j] (sel NULL: j); d >= 2 by banded contractions.
fgr_status run_decompose_tensor(fgr_ctx *ctx, const AxisDev *axes, const void *u_dev, int64_t m,
                                const int64_t *sel, double *a, cudaStream_t st, Scratch &scratch);
// FGR_E_INVALID unless every sel[j] (device memory) lies in [0, total); waits
// for the stream.
fgr_status check_selection_device(fgr_ctx *ctx, const int64_t *sel, int64_t m, int64_t total, cudaStream_t st,
                                  Scratch &scratch);
// out = a0 * f, complex, planes [re][m] then [im][m].
fgr_status run_scale_amplitudes(const double *a0, const double *f, double *out, int64_t m, cudaStream_t st);
fgr_status run_direct(fgr_ctx *ctx, const PacketsDev &pk, void *u_dev, cudaStream_t st,
                      Scratch &scratch);
// check_finite: the bounds reduction also tests every packet value and the
// call returns FGR_E_INVALID, before writing anything, if one is not finite.
fgr_status run_fggc(fgr_ctx *ctx, const PacketsDev &pk, void *u_dev, cudaStream_t st,
                    Scratch &scratch, bool check_finite = false);
// Upper bounds of the buffers that a call can do without (fgr_ctx::spare_bytes) and of
// the 3-D FGGC binning, for the server's account: FP32 1-D direct sums of n points
// aiming at target CTAs, FP32 FGGC of m packets in d >= 2 dimensions.
size_t direct1_spare_bytes(int64_t m, int64_t n, int target);
size_t fggc_spare_bytes(int d, int n1, int64_t m);
// Device bytes owned by an FGGC plan (api.cu).
size_t plan_device_bytes(const fgr_fggc_plan *plan);

// n <= 64 requests of one dimension and precision; scratch[r] belongs to request r
fgr_status run_direct_batch(int n, fgr_ctx *const *ctxs, const PacketsDev *pks, void *const *us,
                            cudaStream_t st, Scratch **scratch, Scratch &shared);

// Event-based stage timer (active only when ctx->timing.enabled).
class StageTimer {
  public:
    StageTimer(fgr_ctx *ctx, cudaStream_t s);
    ~StageTimer();
    void mark(double *slot);  // time since the previous mark goes to *slot
    void finish();            // total -> last.total_ms

  private:
    fgr_ctx *ctx_;
    cudaStream_t s_;
    cudaEvent_t ev_[24] = {};
    double *slot_[24] = {};
    int n_ = 0;
};

inline size_t elem_bytes(int precision) { return precision == FGR_FP64 ? 16 : 8; }

int64_t rk4_nsteps(double t, double dt);

}  // namespace fgr
