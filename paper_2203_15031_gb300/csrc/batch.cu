// Batched SPMESL: many independent fits of different p and n in one pass of
// launches over all of them (Gram, standardisation, column order, coordinate descent, Theta).
// With SPMESL_MIXED the Gram of every fit given as X runs as split-BF16
// products on the tensor cores (one batched split/transpose launch, then one
// persistent tcgen05 launch over the tiles of all fits); the rest runs in
// FP32 with sigma and Theta in FP64, as in the single-fit path.  SPMESL_FP64
// does the same with the digit planes of gram_f64.cu.
//
// Every launch covers all fits at once.  Fits are ordered by decreasing p so
// the longest column chains start first.  A descriptor table in the
// workspace gives each fit its buffers and its first global column / tile
// index; a block or warp finds its fit by binary search over those prefix
// sums.  The coordinate-descent launch is one dynamic queue of all columns of
// all fits (one warp per column, the same column solver as spmesl_fit), so a
// fit's slow columns overlap with other fits' work instead of idling the GPU.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <new>
#include <numeric>
#include <vector>

#include "cd_device.cuh"
#include "gram_device.cuh"
#include "gram_f64.cuh"
#include "gram_tc.cuh"

namespace spmesl {

struct BatchFit {
    const void* X;        // device data (n x p, ld p) or nullptr
    const void* S;        // covariance the fit reads (user S or the Gram output)
    void* Sg;             // Gram output in the workspace (when X is given)
    void* mu;             // column means (centring)
    void* SC;
    void* BT;
    void* diag;
    double* cs;
    float* csf;
    double* sigma;
    int* col_status;
    double* Theta;
    double* sigma_out;
    FitCtrl* ctrl;
    void* XhT;            // split-BF16 operands (SPMESL_MIXED with X), or the digit
    void* XlT;            // planes and the columns' exponents (SPMESL_FP64 with X)
    float* cmax;          // first-sweep chunk maxima of the lazy solver (standardised fits)
    double lambda0;
    double diag_eps;      // rounding bound of the working matrix (diagnostics)
    unsigned* rows;       // moved-coordinate bitmap of the fit (opts.count_rows) or nullptr
    double* hand;         // per column the last sigma step at a hand-over (2 doubles); after the
                          // descent 1 / sigma_j^2 in the first
    int* nsup;            // per column the length of its coefficient list (nullptr: dense rows)
    int n, p, ldp;
    int col_start, gram_start, theta_start;
    int split_start;      // first block of the batched split/transpose launch
    int prep_start;       // first block of the standardisation launch
};

thread_local bool g_batch_pageable_staging = false;

struct BatchHeader {
    int next_col;         // column queue of the lazy launch
    int ovf_count;        // columns handed from the lazy kernel to the block solver
    int ovf_next;         // block solver's position in that queue
    int n_heavy;          // heavy columns: the first n_heavy of the heat order
    int heavy_next;       // block solver's position among them
    int pad[59];
};

// Largest f with prefix[f] <= idx (prefix ascending, prefix[0] = 0).
__device__ __forceinline__ int find_fit(const int* __restrict__ prefix, int count, int idx) {
    int lo = 0, hi = count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (prefix[mid] <= idx) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

template <typename T>
__global__ void batch_mean_kernel(const BatchFit* __restrict__ fits) {
    const BatchFit& f = fits[blockIdx.y];
    if (!f.X || !f.mu) return;
    if ((int)blockIdx.x * 32 >= f.p) return;
    column_means<T>(static_cast<const T*>(f.X), f.n, f.p, f.p, static_cast<T*>(f.mu),
                    blockIdx.x * 32);
}

__global__ void __launch_bounds__(GRAM_THREADS) batch_gram_kernel(const BatchFit* __restrict__ fits,
                                                                 const int* __restrict__ gram_prefix,
                                                                 int count) {
    const int fi = find_fit(gram_prefix, count, blockIdx.x);
    const BatchFit& f = fits[fi];
    int tm, tn;
    upper_tile(blockIdx.x - f.gram_start, (f.p + GRAM_BM - 1) / GRAM_BM, tm, tn);
    gram_tile<GRAM_BM, GRAM_BK, GRAM_THREADS, 8, 4, false>(static_cast<const float*>(f.X), f.n, f.p, f.p,
                                           static_cast<const float*>(f.mu),
                                           static_cast<float*>(f.Sg), f.p,
                                           (float)(1.0 / (double)f.n), tm, tn);
}

// Split/transpose of every fit given as X (SPMESL_MIXED): blocks of 64
// samples x 32 columns over each fit's padded sample dimension (a multiple
// of 64) and columns; blockDim 32 x 8.
__global__ void batch_split_kernel(const BatchFit* __restrict__ fits,
                                   const int* __restrict__ split_prefix, int count) {
    const int fi = find_fit(split_prefix, count, blockIdx.x);
    const BatchFit& f = fits[fi];
    const int n_pad = tc_pad_n(f.n);
    const int bx = n_pad / 64;
    const int idx = blockIdx.x - f.split_start;
    split_transpose_tile64(static_cast<const float*>(f.X), f.n, f.p, f.p,
                           static_cast<const float*>(f.mu), static_cast<__nv_bfloat16*>(f.XhT),
                           static_cast<__nv_bfloat16*>(f.XlT), n_pad, (idx % bx) * 64,
                           (idx / bx) * 32);
}

// Exponents and digit planes of every fit given as X (SPMESL_FP64): one block
// of 32 x 8 per 32 columns.
__global__ void __launch_bounds__(256) batch_digits_kernel(const BatchFit* __restrict__ fits,
                                                          const int* __restrict__ split_prefix,
                                                          int count, int* __restrict__ marks, int s0) {
    const int fi = find_fit(split_prefix, count, blockIdx.x);
    const BatchFit& f = fits[fi];
    if (f.n <= s0) return;
    int* expo = static_cast<int*>(f.XlT);
    f64_digit_columns(static_cast<const double*>(f.X), f.n, f.p, f.p,
                      static_cast<const double*>(f.mu), expo, marks + blockIdx.x,
                      f64_counts(expo, f.p), static_cast<__nv_bfloat16*>(f.XhT),
                      (blockIdx.x - f.split_start) * 32, s0);
}

template <typename T>
__global__ void batch_prep_diag_kernel(const BatchFit* __restrict__ fits, int standardize) {
    const BatchFit& f = fits[blockIdx.y];
    const T* S = static_cast<const T*>(f.S);
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < f.p; j += gridDim.x * blockDim.x) {
        const double d = (double)S[(size_t)j * f.p + j];
        if (!(d > 0.0) || !isfinite(d)) set_error(f.ctrl, DEV_ERR_NONFINITE);
        const double c = standardize ? 1.0 / sqrt(d) : 1.0;
        f.cs[j] = c;
        f.csf[j] = (float)c;
        f.sigma[j] = 1.0;
        f.col_status[j] = COL_OK;
    }
}

// The heat order of a batch's columns (decreasing heat, ties in any order:
// a column's result does not depend on when it runs) as a counting sort over
// ORDER_BLOCKS blocks: per-block bin counts, then each (bin, block) pair's
// first position (bins in decreasing heat, blocks in turn), then the scatter.
constexpr int ORDER_BLOCKS = 128;
__global__ void __launch_bounds__(256) heat_hist_kernel(const int* __restrict__ heat, int n,
                                                        int* __restrict__ hist) {
    __shared__ int bin[HEAT_BINS];
    for (int t = threadIdx.x; t < HEAT_BINS; t += blockDim.x) bin[t] = 0;
    __syncthreads();
    const int chunk = (n + gridDim.x - 1) / gridDim.x;
    const int lo = blockIdx.x * chunk, hi = min(n, lo + chunk);
    for (int i = lo + threadIdx.x; i < hi; i += blockDim.x)
        atomicAdd(&bin[min(heat[i], HEAT_BINS - 1)], 1);
    __syncthreads();
    for (int t = threadIdx.x; t < HEAT_BINS; t += blockDim.x) hist[blockIdx.x * HEAT_BINS + t] = bin[t];
}

// One block of HEAT_BINS threads: hist[b][h] becomes the first position of
// block b's columns of heat h; *n_heavy (if given) the count of heat above
// heavy_heat.
__global__ void heat_offsets_kernel(int* __restrict__ hist, int nblocks, int* __restrict__ n_heavy,
                                    int heavy_heat) {
    __shared__ int total[HEAT_BINS];
    const int h = threadIdx.x;
    int t = 0;
    for (int b = 0; b < nblocks; ++b) t += hist[b * HEAT_BINS + h];
    total[h] = t;
    __syncthreads();
    int run = 0;
    for (int g = HEAT_BINS - 1; g > h; --g) run += total[g];
    if (n_heavy && h == heavy_heat) *n_heavy = run;
    for (int b = 0; b < nblocks; ++b) {
        const int v = hist[b * HEAT_BINS + h];
        hist[b * HEAT_BINS + h] = run;
        run += v;
    }
}

__global__ void __launch_bounds__(256) heat_scatter_kernel(const int* __restrict__ heat, int n,
                                                           const int* __restrict__ hist,
                                                           int* __restrict__ order) {
    __shared__ int cur[HEAT_BINS];
    for (int t = threadIdx.x; t < HEAT_BINS; t += blockDim.x) cur[t] = hist[blockIdx.x * HEAT_BINS + t];
    __syncthreads();
    const int chunk = (n + gridDim.x - 1) / gridDim.x;
    const int lo = blockIdx.x * chunk, hi = min(n, lo + chunk);
    for (int i = lo + threadIdx.x; i < hi; i += blockDim.x)
        order[atomicAdd(&cur[min(heat[i], HEAT_BINS - 1)], 1)] = i;
}

// One warp per row, PREP_ROWS rows per block, the block's rows all of one
// fit (found from the block prefix), so every block has the same work whatever
// the fit sizes; same arithmetic as the single-fit prep_matrix_kernel (BT
// needs no clearing: every solver writes its whole row).  With heat, also
// counts per column the off-diagonal entries of the standardised matrix
// above lambda0: the coordinates that can move in the column's first sweep,
// a predictor of how long the column takes.  In fits below heavy_min_p columns the count is
// capped at heavy_heat, so none of their columns is routed to the block
// solver by heat (the single-fit rule).
constexpr int PREP_ROWS = 8;
template <typename T>
__global__ void __launch_bounds__(32 * PREP_ROWS) batch_prep_matrix_kernel(
    const BatchFit* __restrict__ fits, const int* __restrict__ prep_prefix, int count,
    int* __restrict__ heat, int heavy_heat, int heavy_min_p) {
    const int fi = find_fit(prep_prefix, count, blockIdx.x);
    const BatchFit& f = fits[fi];
    const int lane = threadIdx.x & 31;
    const int r = (blockIdx.x - f.prep_start) * PREP_ROWS + (int)(threadIdx.x >> 5);
    if (r >= f.p) return;                      // warp-uniform
    int cnt = 0;
    float top = 0.f;
    const bool bad = standardize_row<T>(static_cast<const T*>(f.S), f.p, f.ldp, r, f.cs, f.csf,
                                        static_cast<T*>(f.SC), nullptr,
                                        static_cast<T*>(f.diag), lane, 32, (T)f.lambda0,
                                        heat ? &cnt : nullptr, f.cmax, &top);
    if (f.cmax && lane == 0) static_cast<T*>(f.diag)[r] = (T)top;
    if (heat) {
        cnt = __reduce_add_sync(FULL_MASK, cnt);
        if (lane == 0) heat[f.col_start + r] = min(cnt, f.p >= heavy_min_p ? INT_MAX : heavy_heat);
    }
    if (__any_sync(FULL_MASK, bad) && lane == 0) set_error(f.ctrl, DEV_ERR_NONFINITE);
}

template <typename T>
__device__ __forceinline__ CDArgs<T> column_args(const BatchFit& f, double tol, float tolf,
                                                 int maxit, int ovf_supp = LAZY_CAP) {
    CDArgs<T> a;
    a.SC = static_cast<const T*>(f.SC);
    a.BT = static_cast<T*>(f.BT);
    a.GT = nullptr;
    a.diag = static_cast<const T*>(f.diag);
    a.sigma = f.sigma;
    a.col_status = f.col_status;
    a.active = a.active_next = a.flag = nullptr;
    a.ctrl = f.ctrl;
    a.p = f.p;
    a.ldp = f.ldp;
    a.maxit = maxit;
    a.lambda0 = f.lambda0;
    a.tol = tol;
    a.tolf = tolf;
    a.ovf_list = nullptr;
    a.ovf_count = nullptr;
    a.order = nullptr;
    a.n_queue = f.p;
    a.ovf_supp = ovf_supp;
    a.chunk_max = f.cmax;
    a.rows_moved = f.rows;
    a.rows_words = rows_words(f.p);
    a.hand = f.hand;
    a.nsup = f.nsup;
    a.Theta = f.nsup ? f.Theta : nullptr;
    return a;
}

// Distinct moved coordinates of every fit (opts.count_rows): one block per fit.
__global__ void batch_rows_count_kernel(const BatchFit* __restrict__ fits) {
    const BatchFit& f = fits[blockIdx.x];
    if (f.rows)
        count_rows_moved(f.rows, rows_bitmap_bytes(f.p) / 4, f.ctrl, threadIdx.x, blockDim.x);
}

// Eager gradient over all columns of all fits.
template <typename T, bool STD>
__global__ void __launch_bounds__(512) batch_cd_kernel(const BatchFit* __restrict__ fits,
                                                       const int* __restrict__ col_prefix,
                                                       int count, int total_cols, int max_ldp,
                                                       double tol, float tolf, int maxit,
                                                       BatchHeader* hdr) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    T* g = reinterpret_cast<T*>(smem_raw + (size_t)warp * warp_smem_bytes<T>(max_ldp));
    for (;;) {
        int gc = 0;
        if (lane == 0) gc = atomicAdd(&hdr->next_col, 1);
        gc = __shfl_sync(FULL_MASK, gc, 0);
        if (gc >= total_cols) break;
        const int fi = find_fit(col_prefix, count, gc);
        const BatchFit& f = fits[fi];
        if (*reinterpret_cast<volatile int*>(&f.ctrl->err) != 0) continue;
        const CDArgs<T> a = column_args<T>(f, tol, tolf, maxit);
        T* b = g + f.ldp;
        int* list = reinterpret_cast<int*>(b + f.ldp);
        ColCounters cnt;
        solve_column<T, STD>(gc - f.col_start, g, b, list, a, cnt);
        flush_counters(f.ctrl, cnt);
    }
}

constexpr int PREFIX_SMEM = 1024;

// Lazy gradient over all columns of all fits; overflowing columns are queued
// for the block solver, and the first n_heavy columns of the heat order
// belong to it from the start.
// At most 8 warps a block; MINB blocks an SM.  Three (80 registers) carry most
// columns a second; two (128 registers) solve one column sooner, with more of its
// loads in flight and no spills, which decides while the longest columns do, and in FP64,
// where 80 registers spill most.  How long that is depends on the networks too; by
// sizes, a batch of unlike fits, whose longest columns are longer than the mean, has
// two up to LAZY_WIDE_MIXED columns per resident warp of that form (45: 109440 on 152
// SMs), one of like fits up to LAZY_WIDE_COLS (14: 34048).  A whole pass in ms, two and three:
// fits of p 50 to 2000, 128 (62 k columns) 1.03 and 1.20, 200 (98 k) 1.41 and 1.47, 256
// (133 k) 1.90 and 1.81; Erdos-Renyi p = 2000, 14 fits (28 k) 0.466 and 0.505, 20 (40 k)
// 0.629 and 0.614, 40 (80 k) 1.21 and 1.15; p = 500, 80 (40 k) 0.457 and 0.441.  Left on the
// slower side: AR(1) p = 2000, 10 fits (20 k) 0.491 and 0.468; p = 4000, 12 (48 k) 1.05
// and 1.09.
constexpr int LAZY_MAX_WARPS = 8;
constexpr int LAZY_WIDE_COLS = 14, LAZY_WIDE_MIXED = 45;
template <typename T, bool STD, int MINB>
__global__ void __launch_bounds__(32 * LAZY_MAX_WARPS, MINB) batch_cd_lazy_kernel(const BatchFit* __restrict__ fits,
                                                            const int* __restrict__ col_prefix,
                                                            int count, int total_cols, int max_ldp,
                                                            double tol, float tolf, int maxit,
                                                            BatchHeader* hdr, int* ovf_list,
                                                            const int* __restrict__ order,
                                                            int ovf_supp) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // the column prefix in shared memory: every column starts with a search of it
    __shared__ int sprefix[PREFIX_SMEM];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    unsigned char* wsm = smem_raw + (size_t)warp * lazy_warp_smem_bytes<T>(max_ldp);
    const int q0 = order ? *reinterpret_cast<volatile int*>(&hdr->n_heavy) : 0;
    const bool sp = count < PREFIX_SMEM;
    if (sp)
        for (int i = threadIdx.x; i <= count; i += blockDim.x) sprefix[i] = col_prefix[i];
    __syncthreads();
    const int* __restrict__ prefix = sp ? sprefix : col_prefix;
    for (;;) {
        int gc = 0;
        if (lane == 0) {
            gc = q0 + atomicAdd(&hdr->next_col, 1);
            if (order && gc < total_cols) gc = order[gc];
        }
        gc = __shfl_sync(FULL_MASK, gc, 0);
        if (gc >= total_cols) break;
        const int fi = find_fit(prefix, count, gc);
        const BatchFit& f = fits[fi];
        if (*reinterpret_cast<volatile int*>(&f.ctrl->err) != 0) continue;
        const CDArgs<T> a = column_args<T>(f, tol, tolf, maxit, ovf_supp);
        ColCounters cnt;
        if (!solve_column_lazy<T, STD>(gc - f.col_start, wsm, a, cnt) && lane == 0)
            ovf_list[atomicAdd(&hdr->ovf_count, 1)] = gc;
        __syncwarp();
        flush_counters(f.ctrl, cnt);
    }
}

// Block solver over the heavy columns at the head of the heat order
// (from_overflow = 0, beside the lazy launch) or over the columns the lazy
// launch handed over (from_overflow = 1, after it); one block per column.
template <typename T, bool STD>
__global__ void __launch_bounds__(BLK_THREADS, 1) batch_cd_block_kernel(const BatchFit* __restrict__ fits,
                                                                     const int* __restrict__ col_prefix,
                                                                     int count, double tol, float tolf, int maxit,
                                                                     BatchHeader* hdr,
                                                                     const int* __restrict__ queue,
                                                                     int from_overflow) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ BlockScratch sc;
    const int nq = from_overflow ? *reinterpret_cast<volatile int*>(&hdr->ovf_count)
                                 : *reinterpret_cast<volatile int*>(&hdr->n_heavy);
    int* next = from_overflow ? &hdr->ovf_next : &hdr->heavy_next;
    for (;;) {
        if (threadIdx.x == 0) {
            const int t = atomicAdd(next, 1);
            sc.col = t < nq ? queue[t] : -1;
        }
        __syncthreads();
        const int gc = sc.col;
        __syncthreads();
        if (gc < 0) break;
        const int fi = find_fit(col_prefix, count, gc);
        const BatchFit& f = fits[fi];
        if (*reinterpret_cast<volatile int*>(&f.ctrl->err) != 0) continue;
        const CDArgs<T> a = column_args<T>(f, tol, tolf, maxit);
        ColCounters cnt;
        solve_column_block<T, STD>(gc - f.col_start, smem_raw, a, cnt, sc);
        flush_counters_block(f.ctrl, cnt);
    }
}

// Optimality diagnostics of every column of every fit (opts.diagnostics):
// one block per column, grid-stride over the columns.
template <typename T>
__global__ void __launch_bounds__(32 * DIAG_WARPS) batch_diag_kernel(
    const BatchFit* __restrict__ fits, const int* __restrict__ col_prefix, int count,
    int total_cols) {
    __shared__ DiagShared sh;
    for (int gc = blockIdx.x; gc < total_cols; gc += gridDim.x) {
        const int fi = find_fit(col_prefix, count, gc);
        const BatchFit& f = fits[fi];
        if (*reinterpret_cast<volatile int*>(&f.ctrl->err) != 0) continue;   // block-uniform
        const CDArgs<T> a = column_args<T>(f, 0.0, 0.f, 1);
        DiagMax d;
        diagnose_column<T>(gc - f.col_start, sh, a, f.diag_eps, d);
        flush_diag(f.ctrl, d);
        __syncthreads();
    }
}

template <typename T>
__global__ void batch_theta_kernel(const BatchFit* __restrict__ fits,
                                   const int* __restrict__ theta_prefix, int count) {
    const int fi = find_fit(theta_prefix, count, blockIdx.x);
    const BatchFit& f = fits[fi];
    if (*reinterpret_cast<volatile int*>(&f.ctrl->err) != 0) return;
    theta_pair<T>(static_cast<const T*>(f.BT), f.p, f.ldp, f.sigma, f.cs, f.Theta, f.sigma_out,
                  f.ctrl, blockIdx.x - f.theta_start);
}

// The last step of sigma_j's square root (sqrt_last) and 1 / sigma_j^2 of every column, one
// per lane: an FP64 division takes a warp some 250 cycles of the FP64 pipe whatever its
// active lanes, so the lists' pass below reads it.
__global__ void __launch_bounds__(256) batch_inv_kernel(const BatchFit* __restrict__ fits) {
    const BatchFit& f = fits[blockIdx.y];
    if (*reinterpret_cast<volatile int*>(&f.ctrl->err) != 0) return;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < f.p; j += gridDim.x * blockDim.x) {
        const double s = sqrt_last(f.hand[2 * (size_t)j + 1], f.sigma[j]);
        f.sigma[j] = s;
        f.hand[2 * (size_t)j] = 1.0 / (s * s);
    }
}

// Theta's nonzero entries after the column solvers (see theta_column), the
// block's columns all of one fit.
constexpr int THETA_COLS = 256 / THETA_LANES;
template <typename T>
__global__ void __launch_bounds__(256) batch_theta_list_kernel(const BatchFit* __restrict__ fits,
                                                              const int* __restrict__ theta_prefix,
                                                              int count) {
    const int fi = find_fit(theta_prefix, count, blockIdx.x);
    const BatchFit& f = fits[fi];
    if (*reinterpret_cast<volatile int*>(&f.ctrl->err) != 0) return;
    const int j = (blockIdx.x - f.theta_start) * THETA_COLS + (int)threadIdx.x / THETA_LANES;
    const double* __restrict__ inv = f.hand;
    unsigned nnz = 0;
    if (j < f.p)
        nnz = theta_column<T>(static_cast<const T*>(f.BT), f.nsup, f.p, f.ldp, j, f.sigma, f.cs,
                              f.Theta, f.sigma_out, [&](int k) { return inv[2 * (size_t)k]; });
    nnz = __reduce_add_sync(FULL_MASK, nnz);
    if ((threadIdx.x & 31) == 0 && nnz) atomicAdd(&f.ctrl->nnz, (unsigned long long)nnz);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
namespace {

struct FitPlan {
    int src;                 // index in the caller's array
    int n, p, ldp;
    double lambda0;
    const void* X;
    const void* S;
    double* Theta;
    double* sigma;
    size_t off_ctrl, off_cs, off_csf, off_sigma, off_status, off_diag, off_cmax, off_mu, off_Sg, off_SC,
        off_BT, off_rows, off_hand;
    size_t off_XhT, off_XlT;
    int col_start, gram_start, theta_start, split_start, prep_start;
};

int num_sms() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 1;
    }
    return sms;
}

int max_smem_block() {
    static int v = 0;
    if (!v) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    }
    return v;
}

}  // namespace
}  // namespace spmesl

using namespace spmesl;

struct spmesl_batch {
    int count = 0;
    int precision = SPMESL_FP32;
    int standardize = 1;
    int center = 0;
    int use_graph = 0;
    double tol = 1e-6;
    int maxit = 1000;
    int warps_per_block = 0;       // 0 = automatic
    int gradient = SPMESL_GRADIENT_AUTO;
    int heavy_heat = 0, heavy_min_p = 0;   // routing limits of spmesl_opts (0: defaults)
    int diagnostics = 0;           // optimality diagnostics after the coordinate descent
    int handover = 0;              // the lazy solver's hand-over support (0: default)
    mutable std::vector<spmesl_stats> fit_stats;   // per fit, caller's order (last result)
    size_t off_ovf = 0;            // queue of columns for the eager launch (total_cols ints)
    size_t off_heat = 0, off_order = 0;   // per-column heat and the lazy queue's order
    size_t off_hist = 0;                  // the heat order's per-block bin counts
    std::vector<FitPlan> plan;     // ordered by decreasing p
    size_t off_hdr = 0, off_desc = 0, off_colp = 0, off_gramp = 0, off_thetap = 0, off_ctrls = 0;
    size_t off_prepp = 0;          // block prefix of the standardisation launch
    int total_prep = 0;
    int count_rows = 0;            // moved-coordinate bitmaps (measurement)
    size_t off_rows = 0, rows_bytes = 0;   // all fits' bitmaps, contiguous
    // SPMESL_MIXED, SPMESL_FP64: tensor-core Gram table, fit of every tile, split prefixes
    size_t off_tcfit = 0, off_tilefit = 0, off_splitp = 0;
    int total_split = 0;
    // SPMESL_FP64: marks of the columns that the Gram does not scale, and their blocks
    size_t off_marks = 0;
    int total_direct = 0, max_nx = 1;   // largest n of the fits given as X
    size_t ws_bytes = 0;
    int total_cols = 0, total_gram = 0, total_theta = 0, max_ldp = 32, max_p = 2, max_n = 1;
    bool any_x = false;
    // pinned staging of the descriptor table and the prefix arrays
    unsigned char* pinned = nullptr;
    bool pinned_is_pageable = false;
    size_t table_bytes = 0;
    const void* table_ws = nullptr;    // workspace the staged table points into
    cudaGraphExec_t graph = nullptr;
    const void* graph_ws = nullptr;
    int graph_W = -1;
    int graph_key[3] = {0, 0, 0};   // handover, heavy_min_p, heavy_heat of the captured graph
    cudaStream_t cap_stream = nullptr;
    // side stream: the block solver's launch over the heavy columns
    cudaStream_t side2 = nullptr;
    cudaEvent_t fork2 = nullptr, join2 = nullptr;
    // record_phase_times (runs without a graph): events around the CD launch
    int record_phase_times = 0;
    cudaEvent_t ev[2] = {nullptr, nullptr};
    bool ev_recorded = false;
};

namespace {

// Columns per resident warp up to which the lazy kernel runs two blocks an SM: the fits are
// unlike when the largest has 1.5 times the chunks of the mean column's.
int lazy_wide_cols(const spmesl_batch* b) {
    long long chunks = 0;
    for (const FitPlan& f : b->plan) chunks += (long long)f.p * row_chunks(f.ldp);
    return 2ll * row_chunks(b->max_ldp) * b->total_cols >= 3 * chunks ? LAZY_WIDE_MIXED : LAZY_WIDE_COLS;
}

template <typename T>
cudaError_t enqueue_batch(spmesl_batch* b, unsigned char* ws, cudaStream_t st, int W) {
    const BatchFit* fits = reinterpret_cast<const BatchFit*>(ws + b->off_desc);
    const int* colp = reinterpret_cast<const int*>(ws + b->off_colp);
    const int* gramp = reinterpret_cast<const int*>(ws + b->off_gramp);
    const int* thetap = reinterpret_cast<const int*>(ws + b->off_thetap);
    BatchHeader* hdr = reinterpret_cast<BatchHeader*>(ws + b->off_hdr);
    cudaError_t e;
    // descriptor table + prefix arrays, then the control blocks and the queue
    if ((e = cudaMemcpyAsync(ws + b->off_desc, b->pinned, b->table_bytes, cudaMemcpyHostToDevice,
                             st)) != cudaSuccess)
        return e;
    if ((e = cudaMemsetAsync(ws + b->off_hdr, 0, sizeof(BatchHeader), st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ws + b->off_ctrls, 0, (size_t)256 * b->count, st)) != cudaSuccess)
        return e;
    if (b->count_rows &&
        (e = cudaMemsetAsync(ws + b->off_rows, 0, b->rows_bytes, st)) != cudaSuccess)
        return e;
    const int count = b->count;
    if (b->any_x) {
        if (b->center)
            batch_mean_kernel<T><<<dim3((b->max_p + 31) / 32, count), dim3(32, MEAN_GROUPS), 0, st>>>(
                fits);
        if (b->precision == SPMESL_MIXED) {
            batch_split_kernel<<<b->total_split, dim3(32, 8), 0, st>>>(
                fits, reinterpret_cast<const int*>(ws + b->off_splitp), count);
            if ((e = launch_gram_tc_batch(reinterpret_cast<const TcFit*>(ws + b->off_tcfit),
                                          reinterpret_cast<const int*>(ws + b->off_tilefit),
                                          b->total_gram, st)) != cudaSuccess)
                return e;
        } else if constexpr (sizeof(T) == 8) {
            for (long long s = 0; s < b->max_nx; s += F64_SLAB) {
                const int s0 = (int)s;
                batch_digits_kernel<<<b->total_split, dim3(32, 8), 0, st>>>(
                    fits, reinterpret_cast<const int*>(ws + b->off_splitp), count,
                    reinterpret_cast<int*>(ws + b->off_marks), s0);
                const F64Batch g{reinterpret_cast<const F64Fit*>(ws + b->off_tcfit),
                                 reinterpret_cast<const int*>(ws + b->off_tilefit),
                                 reinterpret_cast<const int*>(ws + b->off_marks), count, b->total_gram,
                                 b->total_split, b->total_direct, s0};
                if ((e = launch_gram_f64_batch(g, st)) != cudaSuccess) return e;
            }
        } else {
            batch_gram_kernel<<<b->total_gram, GRAM_THREADS, 0, st>>>(fits, gramp, count);
        }
    }
    batch_prep_diag_kernel<T><<<dim3((b->max_p + 255) / 256, count), 256, 0, st>>>(fits,
                                                                                   b->standardize);
    // column order for the lazy launch (standardised working matrix only);
    // with AUTO the heavy columns lead it and go to the block solver
    const bool lazy_order = b->gradient != SPMESL_GRADIENT_EAGER && b->standardize;
    const bool route = b->gradient == SPMESL_GRADIENT_AUTO;
    // (the heavy launch only where some fit is large enough to route by heat)
    const bool heavy = route && lazy_order && b->max_p >= heavy_min_p_of(b->heavy_min_p);
    int* heat = reinterpret_cast<int*>(ws + b->off_heat);
    int* order = reinterpret_cast<int*>(ws + b->off_order);
    const int hheat = heavy_heat_of(b->heavy_heat);
    batch_prep_matrix_kernel<T><<<b->total_prep, 256, 0, st>>>(
        fits, reinterpret_cast<const int*>(ws + b->off_prepp), count, lazy_order ? heat : nullptr,
        hheat, heavy_min_p_of(b->heavy_min_p));
    if (lazy_order) {
        int* hist = reinterpret_cast<int*>(ws + b->off_hist);
        heat_hist_kernel<<<ORDER_BLOCKS, 256, 0, st>>>(heat, b->total_cols, hist);
        heat_offsets_kernel<<<1, HEAT_BINS, 0, st>>>(hist, ORDER_BLOCKS,
                                                    heavy ? &hdr->n_heavy : nullptr, hheat);
        heat_scatter_kernel<<<ORDER_BLOCKS, 256, 0, st>>>(heat, b->total_cols, hist, order);
    }

    const float tolf = float_at_least(b->tol);
    const size_t budget = (size_t)max_smem_block() - 1024;
    const bool lazy = b->gradient != SPMESL_GRADIENT_EAGER;
    int* ovf = reinterpret_cast<int*>(ws + b->off_ovf);
    const bool timed = b->record_phase_times && b->ev[0];
    if (timed) cudaEventRecord(b->ev[0], st);
    if (lazy) {
        // block solver: persistent grid, one block per column
        auto bk = b->standardize ? batch_cd_block_kernel<T, true> : batch_cd_block_kernel<T, false>;
        const size_t bsm = block_smem_bytes<T>(b->max_ldp);
        if (bsm > budget) return cudaErrorInvalidValue;
        if ((e = cudaFuncSetAttribute(bk, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)bsm)) != cudaSuccess)
            return e;
        int bper_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bper_sm, bk, BLK_THREADS, bsm)) !=
            cudaSuccess)
            return e;
        const int bgrid = num_sms() * std::max(1, std::min(bper_sm, 2));
        if (heavy) {
            // the heavy columns start first, on the side stream, beside the lazy launch
            if ((e = cudaEventRecord(b->fork2, st)) != cudaSuccess ||
                (e = cudaStreamWaitEvent(b->side2, b->fork2, 0)) != cudaSuccess)
                return e;
            bk<<<bgrid, BLK_THREADS, bsm, b->side2>>>(fits, colp, count, b->tol, tolf, b->maxit, hdr,
                                                      order, 0);
            if ((e = cudaEventRecord(b->join2, b->side2)) != cudaSuccess) return e;
        }
        // W (tuned) shapes the lazy launch, which does almost all the work
        const size_t lper = lazy_warp_smem_bytes<T>(b->max_ldp);
        const int LW = std::max(1, std::min({W, LAZY_MAX_WARPS, (int)(budget / lper)}));
        const size_t lsm = lper * LW;
        auto lk = b->standardize ? batch_cd_lazy_kernel<T, true, 2> : batch_cd_lazy_kernel<T, false, 2>;
        if constexpr (sizeof(T) == 4)
            if (b->total_cols > lazy_wide_cols(b) * num_sms() * 2 * LAZY_MAX_WARPS)
                lk = b->standardize ? batch_cd_lazy_kernel<T, true, 3> : batch_cd_lazy_kernel<T, false, 3>;
        if ((e = cudaFuncSetAttribute(lk, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)lsm)) != cudaSuccess)
            return e;
        int lper_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&lper_sm, lk, 32 * LW, lsm)) !=
            cudaSuccess)
            return e;
        lper_sm = std::max(lper_sm, 1);
        const int lgrid = std::min((b->total_cols + LW - 1) / LW, num_sms() * lper_sm);
        lk<<<lgrid, 32 * LW, lsm, st>>>(fits, colp, count, b->total_cols, b->max_ldp, b->tol, tolf,
                                        b->maxit, hdr, ovf, lazy_order ? order : nullptr,
                                        route ? handover_of(b->handover) : LAZY_CAP);
        // the columns the lazy launch handed over
        bk<<<bgrid, BLK_THREADS, bsm, st>>>(fits, colp, count, b->tol, tolf, b->maxit, hdr, ovf, 1);
        if (heavy && (e = cudaStreamWaitEvent(st, b->join2, 0)) != cudaSuccess) return e;
    } else {
        // eager gradient for every column
        const size_t per_warp = warp_smem_bytes<T>(b->max_ldp);
        const int wmax = (int)std::min<size_t>(16, budget / per_warp);
        if (wmax < 1) return cudaErrorInvalidValue;
        const int EW = std::max(1, std::min(W, wmax));
        const size_t smem = per_warp * EW;
        auto kern = b->standardize ? batch_cd_kernel<T, true> : batch_cd_kernel<T, false>;
        if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem)) != cudaSuccess)
            return e;
        int per_sm = 0;
        if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * EW, smem)) !=
            cudaSuccess)
            return e;
        per_sm = std::max(per_sm, 1);
        const int grid = std::min((b->total_cols + EW - 1) / EW, num_sms() * per_sm);
        kern<<<grid, 32 * EW, smem, st>>>(fits, colp, count, b->total_cols, b->max_ldp, b->tol, tolf,
                                          b->maxit, hdr);
    }
    if (timed) cudaEventRecord(b->ev[1], st);
    if (b->count_rows) batch_rows_count_kernel<<<count, 256, 0, st>>>(fits);
    if (lazy) batch_inv_kernel<<<dim3((b->max_p + 255) / 256, count), 256, 0, st>>>(fits);
    if (b->diagnostics) {
        const int dgrid = std::max(1, std::min(b->total_cols, num_sms() * 16));
        batch_diag_kernel<T><<<dgrid, 32 * DIAG_WARPS, 0, st>>>(fits, colp, count, b->total_cols);
    }
    if (lazy) {
        batch_theta_list_kernel<T><<<b->total_theta, 256, 0, st>>>(fits, thetap, count);
    } else {
        batch_theta_kernel<T><<<b->total_theta, dim3(32, 8), 0, st>>>(fits, thetap, count);
    }
    return cudaGetLastError();
}

// Default warps per block: fill every SM with enough warps for the columns,
// keeping shared memory near half of the SM (see the single-fit launcher).
int auto_warps(const spmesl_batch* b) {
    if (b->gradient != SPMESL_GRADIENT_EAGER) return 8;    // lazy launch: 8 warps per block
    const size_t per_warp = b->precision == SPMESL_FP64 ? warp_smem_bytes<double>(b->max_ldp)
                                                        : warp_smem_bytes<float>(b->max_ldp);
    const size_t budget = (size_t)max_smem_block() - 1024;
    int W = (b->total_cols + num_sms() - 1) / num_sms();
    W = std::min(W, (int)std::max<size_t>(1, (budget / 2) / per_warp));
    return std::max(1, std::min(16, W));
}

// Fill the pinned table with device addresses inside `ws`.
bool stage_table(spmesl_batch* b, unsigned char* ws) {
    BatchFit* t = reinterpret_cast<BatchFit*>(b->pinned);
    const bool mixed = b->precision == SPMESL_MIXED;
    const bool f64 = b->precision == SPMESL_FP64;
    const bool tc = mixed || f64;             // Gram on the tensor cores
    TcFit* tcf = mixed ? reinterpret_cast<TcFit*>(b->pinned + (b->off_tcfit - b->off_desc)) : nullptr;
    F64Fit* dgf = f64 ? reinterpret_cast<F64Fit*>(b->pinned + (b->off_tcfit - b->off_desc)) : nullptr;
    int* tilefit = tc ? reinterpret_cast<int*>(b->pinned + (b->off_tilefit - b->off_desc)) : nullptr;
    int* splitp = tc ? reinterpret_cast<int*>(b->pinned + (b->off_splitp - b->off_desc)) : nullptr;
    int* colp = reinterpret_cast<int*>(b->pinned + (b->off_colp - b->off_desc));
    int* gramp = reinterpret_cast<int*>(b->pinned + (b->off_gramp - b->off_desc));
    int* thetap = reinterpret_cast<int*>(b->pinned + (b->off_thetap - b->off_desc));
    int* prepp = reinterpret_cast<int*>(b->pinned + (b->off_prepp - b->off_desc));
    for (int i = 0; i < b->count; ++i) {
        const FitPlan& f = b->plan[i];
        BatchFit d{};
        d.X = f.X;
        d.Sg = f.X ? ws + f.off_Sg : nullptr;
        d.S = f.X ? d.Sg : f.S;
        d.mu = (f.X && b->center) ? ws + f.off_mu : nullptr;
        d.SC = ws + f.off_SC;
        d.BT = ws + f.off_BT;
        d.diag = ws + f.off_diag;
        // first-sweep chunk maxima: the lazy solver on the standardised matrix
        d.cmax = (b->gradient != SPMESL_GRADIENT_EAGER && b->standardize)
                     ? reinterpret_cast<float*>(ws + f.off_cmax) : nullptr;
        d.cs = reinterpret_cast<double*>(ws + f.off_cs);
        d.csf = reinterpret_cast<float*>(ws + f.off_csf);
        d.sigma = reinterpret_cast<double*>(ws + f.off_sigma);
        d.col_status = reinterpret_cast<int*>(ws + f.off_status);
        d.XhT = (tc && f.X) ? ws + f.off_XhT : nullptr;
        d.XlT = (tc && f.X) ? ws + f.off_XlT : nullptr;
        d.Theta = f.Theta;
        d.sigma_out = f.sigma;
        d.ctrl = reinterpret_cast<FitCtrl*>(ws + f.off_ctrl);
        d.lambda0 = f.lambda0;
        d.diag_eps = diag_eps_for(b->precision, f.X ? f.n : 1);
        d.rows = b->count_rows ? reinterpret_cast<unsigned*>(ws + f.off_rows) : nullptr;
        d.hand = reinterpret_cast<double*>(ws + f.off_hand);
        // the heat counts are dead once the columns are ordered
        d.nsup = b->gradient != SPMESL_GRADIENT_EAGER
                     ? reinterpret_cast<int*>(ws + b->off_heat) + f.col_start : nullptr;
        d.n = f.n;
        d.p = f.p;
        d.ldp = f.ldp;
        d.col_start = f.col_start;
        d.gram_start = f.gram_start;
        d.theta_start = f.theta_start;
        d.prep_start = f.prep_start;
        d.split_start = f.split_start;
        t[i] = d;
        if (mixed) {
            splitp[i] = f.split_start;
            if (f.X) {
                if (!tc_encode_fit(tcf[i], d.XhT, d.XlT, f.n, f.p, static_cast<float*>(d.Sg), f.p,
                                   f.gram_start, TC_BATCH_BN))
                    return false;
                const int nt = tcf[i].g.count();
                for (int k = 0; k < nt; ++k) tilefit[f.gram_start + k] = i;
            } else {
                tcf[i] = TcFit{};
                tcf[i].tile_start = f.gram_start;
            }
        }
        if (f64) {
            splitp[i] = f.split_start;
            if (f.X) {
                if (!f64_encode_fit(dgf[i], static_cast<const double*>(f.X), f.n, f.p, f.p,
                                    static_cast<const double*>(d.mu), static_cast<const int*>(d.XlT),
                                    reinterpret_cast<const int*>(ws + b->off_marks) + f.split_start,
                                    d.XhT, static_cast<double*>(d.Sg), f.p, f.gram_start))
                    return false;
                const int nt = dgf[i].g.count();
                for (int k = 0; k < nt; ++k) tilefit[f.gram_start + k] = i;
            } else {
                dgf[i] = F64Fit{};
                dgf[i].tile_start = f.gram_start;
            }
        }
        colp[i] = f.col_start;
        gramp[i] = f.gram_start;
        thetap[i] = f.theta_start;
        prepp[i] = f.prep_start;
    }
    colp[b->count] = b->total_cols;
    gramp[b->count] = b->total_gram;
    thetap[b->count] = b->total_theta;
    prepp[b->count] = b->total_prep;
    if (tc) splitp[b->count] = b->total_split;
    b->table_ws = ws;
    return true;
}

spmesl_status status_of(const FitCtrl& c) {
    if (c.err == DEV_ERR_NONFINITE) return SPMESL_ENONFINITE;
    if (c.err == DEV_ERR_TIMEOUT) return SPMESL_ETIMEOUT;
    if (c.n_degenerate > 0) return SPMESL_EDEGENERATE;
    if (c.n_not_converged > 0) return SPMESL_NOT_CONVERGED;
    return SPMESL_OK;
}

}  // namespace

extern "C" {

spmesl_status spmesl_batch_create(const spmesl_problem* probs, int count, double tol, int maxit,
                                  const spmesl_opts* opts, spmesl_batch** out) {
    if (!out) return SPMESL_EINVAL;
    *out = nullptr;
    spmesl_opts o;
    if (opts) o = *opts;
    else spmesl_default_opts(&o);
    if (!probs || count < 1 || !(tol > 0.0) || maxit < 1) return SPMESL_EINVAL;
    if (o.precision != SPMESL_FP64 && o.precision != SPMESL_FP32 && o.precision != SPMESL_MIXED)
        return SPMESL_EINVAL;
    if (o.inner_rule != SPMESL_INNER_COLUMN) return SPMESL_EINVAL;
    const int maxp = max_p_for(o.precision);
    for (int i = 0; i < count; ++i) {
        const spmesl_problem& q = probs[i];
        if (q.p < 2 || q.p > maxp || !q.Theta || !q.sigma || (!q.X && !q.S)) return SPMESL_EINVAL;
        if (q.X && q.n < 1) return SPMESL_EINVAL;
        double lam = q.lambda0;
        if (!(lam > 0.0)) lam = spmesl_lambda(o.lambda_rule, q.n, q.p);
        if (!(lam > 0.0) || !isfinite(lam)) return SPMESL_EINVAL;
    }
    spmesl_batch* b = new (std::nothrow) spmesl_batch();
    if (!b) return SPMESL_ENOMEM;
    b->count = count;
    b->precision = o.precision;
    b->standardize = o.standardize ? 1 : 0;
    b->center = o.center ? 1 : 0;
    b->use_graph = o.use_graph ? 1 : 0;
    b->record_phase_times = o.record_phase_times ? 1 : 0;
    b->warps_per_block = o.warps_per_block;
    b->gradient = o.gradient;
    b->heavy_heat = o.heavy_heat;
    b->heavy_min_p = o.heavy_min_p;
    b->diagnostics = o.diagnostics ? 1 : 0;
    b->count_rows = o.count_rows ? 1 : 0;
    b->handover = o.handover;
    b->tol = tol;
    b->maxit = maxit;
    std::vector<int> order(count);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(),
                     [&](int a, int c) { return probs[a].p > probs[c].p; });
    const size_t s = (size_t)elem_size(o.precision);
    const bool mixed = o.precision == SPMESL_MIXED;
    const bool tc = mixed || o.precision == SPMESL_FP64;
    // tensor-core tiles of the whole batch, for the table sizes
    const int tc_bn = mixed ? TC_BATCH_BN : F64_BN;
    long long tc_tiles = 0;
    if (tc)
        for (int i = 0; i < count; ++i)
            if (probs[i].X) tc_tiles += tc_tile_grid(probs[i].p, tc_bn).count();
    if (tc_tiles > (1ll << 30)) return SPMESL_EINVAL;
    size_t off = 0;
    b->off_hdr = off;   off += align_up(sizeof(BatchHeader), 256);
    b->off_desc = off;  off += align_up(sizeof(BatchFit) * count, 256);
    b->off_colp = off;  off += align_up(sizeof(int) * (count + 1), 256);
    b->off_gramp = off; off += align_up(sizeof(int) * (count + 1), 256);
    b->off_thetap = off; off += align_up(sizeof(int) * (count + 1), 256);
    b->off_prepp = off; off += align_up(sizeof(int) * (count + 1), 256);
    if (tc) {
        b->off_tcfit = off;
        off += align_up((mixed ? sizeof(TcFit) : sizeof(F64Fit)) * count, 256);
        b->off_tilefit = off; off += align_up(sizeof(int) * (size_t)std::max<long long>(tc_tiles, 1), 256);
        b->off_splitp = off;  off += align_up(sizeof(int) * (count + 1), 256);
    }
    b->table_bytes = off - b->off_desc;
    b->off_ctrls = off; off += (size_t)256 * count;      // one FitCtrl slot per fit
    int cols = 0, gram = 0, theta = 0, split = 0, prep = 0;
    long long direct = 0;
    for (int k = 0; k < count; ++k) {
        const spmesl_problem& q = probs[order[k]];
        FitPlan f{};
        f.src = order[k];
        f.n = q.n;
        f.p = q.p;
        f.ldp = padded_ld(q.p);
        f.lambda0 = q.lambda0 > 0.0 ? q.lambda0 : spmesl_lambda(o.lambda_rule, q.n, q.p);
        f.X = q.X;
        f.S = q.S;
        f.Theta = q.Theta;
        f.sigma = q.sigma;
        const size_t mat = align_up((size_t)f.p * f.ldp * s, 256);
        f.off_ctrl = b->off_ctrls + (size_t)256 * k;
        f.off_cs = off;     off += align_up((size_t)f.p * 8, 256);
        f.off_csf = off;    off += align_up((size_t)f.p * 4, 256);
        f.off_sigma = off;  off += align_up((size_t)f.p * 8, 256);
        f.off_status = off; off += align_up((size_t)f.p * 4, 256);
        f.off_diag = off;   off += align_up((size_t)f.p * s, 256);
        f.off_cmax = off;   off += align_up((size_t)f.p * row_chunks(f.ldp) * 4, 256);
        f.off_hand = off;   off += align_up((size_t)f.p * 16, 256);
        if (q.X) {
            f.off_mu = off;  off += align_up((size_t)f.p * s, 256);
            f.off_Sg = off;  off += align_up((size_t)f.p * f.p * s, 256);
            if (mixed) {
                const size_t half = tc_operand_bytes(f.n, f.p) / 2;
                f.off_XhT = off; off += half;
                f.off_XlT = off; off += half;
            } else if (tc) {
                f.off_XhT = off; off += f64_digit_bytes(f.n, f.p);
                f.off_XlT = off; off += f64_expo_bytes(f.p);
            }
            b->any_x = true;
            b->max_nx = std::max(b->max_nx, f.n);
        }
        f.off_SC = off;     off += mat;
        f.off_BT = off;     off += mat;
        f.col_start = cols;
        cols += f.p;
        f.gram_start = gram;
        f.split_start = split;
        if (q.X && tc) {
            gram += tc_tile_grid(f.p, tc_bn).count();
            split += (mixed ? tc_pad_n(f.n) / 64 : 1) * ((f.p + 31) / 32);
            if (!mixed) direct = std::min<long long>(direct + f64_direct_blocks(f.p), INT_MAX);
        } else if (q.X) {
            const int t = (f.p + GRAM_BM - 1) / GRAM_BM;
            gram += t * (t + 1) / 2;
        }
        f.theta_start = theta;
        f.prep_start = prep;
        prep += (f.p + PREP_ROWS - 1) / PREP_ROWS;
        if (o.gradient != SPMESL_GRADIENT_EAGER) theta += (f.p + THETA_COLS - 1) / THETA_COLS;
        else theta += o.precision == SPMESL_FP64 ? theta_pairs<double>(f.p) : theta_pairs<float>(f.p);
        b->max_ldp = std::max(b->max_ldp, f.ldp);
        b->max_p = std::max(b->max_p, f.p);
        b->max_n = std::max(b->max_n, f.n);
        b->plan.push_back(f);
    }
    b->total_cols = cols;
    b->total_gram = gram;
    b->total_split = split;
    b->total_direct = (int)direct;
    if (tc && !mixed) {
        b->off_marks = off;
        off += align_up(sizeof(int) * (size_t)std::max(split, 1), 256);
    }
    b->total_theta = theta;
    b->total_prep = prep;
    if (b->count_rows) {
        b->off_rows = off;
        for (FitPlan& f : b->plan) {
            f.off_rows = off;
            off += align_up(rows_bitmap_bytes(f.p), 256);
        }
        b->rows_bytes = off - b->off_rows;
    }
    b->off_ovf = off;
    off += align_up(sizeof(int) * (size_t)cols, 256);
    b->off_heat = off;
    off += align_up(sizeof(int) * (size_t)cols, 256);
    b->off_order = off;
    off += align_up(sizeof(int) * (size_t)cols, 256);
    b->off_hist = off;
    off += align_up(sizeof(int) * (size_t)ORDER_BLOCKS * HEAT_BINS, 256);
    b->ws_bytes = off;
    if (spmesl::g_batch_pageable_staging) {
        // used by the serving context: no pinned allocation (whose release can
        // synchronise the device) per admission round
        // (256-byte aligned: the table holds 64-byte aligned tensor maps)
        b->pinned = static_cast<unsigned char*>(std::aligned_alloc(256, align_up(b->table_bytes, 256)));
        b->pinned_is_pageable = true;
        if (!b->pinned) {
            delete b;
            return SPMESL_ENOMEM;
        }
    } else if (cudaMallocHost(&b->pinned, b->table_bytes) != cudaSuccess) {
        delete b;
        return SPMESL_ENOMEM;
    }
    *out = b;
    return SPMESL_OK;
}

size_t spmesl_batch_workspace_bytes(const spmesl_batch* b) { return b ? b->ws_bytes : 0; }

spmesl_status spmesl_batch_run(spmesl_batch* b, void* workspace, size_t ws_bytes, void* stream) {
    if (!b || !workspace || ws_bytes < b->ws_bytes) return SPMESL_EINVAL;
    if (reinterpret_cast<uintptr_t>(workspace) & 255u) return SPMESL_EINVAL;
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (b->table_ws != workspace) {
        // the staged table may still be read by an earlier copy on `st`
        if (b->table_ws && cudaStreamSynchronize(st) != cudaSuccess) return SPMESL_ECUDA;
        if (!stage_table(b, ws)) {
            b->table_ws = nullptr;
            return SPMESL_ECUDA;
        }
    }
    const int W = b->warps_per_block > 0 ? b->warps_per_block : auto_warps(b);
    if (!b->side2) {
        if (cudaStreamCreateWithFlags(&b->side2, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&b->fork2, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&b->join2, cudaEventDisableTiming) != cudaSuccess)
            return SPMESL_ECUDA;
    }
    auto enqueue = [&](cudaStream_t s2) {
        return b->precision == SPMESL_FP64 ? enqueue_batch<double>(b, ws, s2, W)
                                           : enqueue_batch<float>(b, ws, s2, W);
    };
    if (!b->use_graph) {
        if (b->record_phase_times && !b->ev[0]) {
            if (cudaEventCreate(&b->ev[0]) != cudaSuccess || cudaEventCreate(&b->ev[1]) != cudaSuccess)
                return SPMESL_ECUDA;
        }
        cudaError_t e = enqueue(st);
        b->ev_recorded = b->record_phase_times && e == cudaSuccess;
        return e == cudaSuccess ? SPMESL_OK : SPMESL_ECUDA;
    }
    b->ev_recorded = false;
    const int gkey[3] = {b->handover, b->heavy_min_p, b->heavy_heat};
    if (!b->graph || b->graph_ws != workspace || b->graph_W != W ||
        memcmp(gkey, b->graph_key, sizeof(gkey)) != 0) {
        if (b->graph) {
            cudaGraphExecDestroy(b->graph);
            b->graph = nullptr;
        }
        if (!b->cap_stream &&
            cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking) != cudaSuccess)
            return SPMESL_ECUDA;
        cudaGraph_t graph = nullptr;
        if (cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
            return SPMESL_ECUDA;
        cudaError_t e = enqueue(b->cap_stream);
        cudaError_t e2 = cudaStreamEndCapture(b->cap_stream, &graph);
        if (e != cudaSuccess || e2 != cudaSuccess) {
            if (graph) cudaGraphDestroy(graph);
            return SPMESL_ECUDA;
        }
        e = cudaGraphInstantiate(&b->graph, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return SPMESL_ECUDA;
        b->graph_ws = workspace;
        b->graph_W = W;
        memcpy(b->graph_key, gkey, sizeof(gkey));
    }
    return cudaGraphLaunch(b->graph, st) == cudaSuccess ? SPMESL_OK : SPMESL_ECUDA;
}

spmesl_status spmesl_batch_result(const spmesl_batch* b, const void* workspace, int32_t* statuses,
                                  spmesl_stats* stats, void* stream) {
    if (!b || !workspace) return SPMESL_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (cudaStreamSynchronize(st) != cudaSuccess) return SPMESL_ECUDA;
    const unsigned char* ws = static_cast<const unsigned char*>(workspace);
    std::vector<unsigned char> ctrls((size_t)256 * b->count);
    if (cudaMemcpyAsync(ctrls.data(), ws + b->off_ctrls, ctrls.size(), cudaMemcpyDeviceToHost,
                        st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return SPMESL_ECUDA;
    spmesl_status worst = SPMESL_OK;
    spmesl_stats agg;
    memset(&agg, 0, sizeof(agg));
    b->fit_stats.assign(b->count, agg);
    for (const FitPlan& f : b->plan) {
        FitCtrl c;
        memcpy(&c, ctrls.data() + (f.off_ctrl - b->off_ctrls), sizeof(c));
        const spmesl_status s = status_of(c);
        if (statuses) statuses[f.src] = s;
        spmesl_stats& fs = b->fit_stats[f.src];
        fs.status = s;
        fs.outer_iters = c.outer_max;
        fs.inner_sweeps = (int64_t)c.total_sweeps;
        fs.moves = (int64_t)c.moves;
        fs.active_sweeps = (int64_t)c.act_sweeps;
        fs.active_moves = (int64_t)c.act_moves;
        fs.nnz_B = (int64_t)c.nnz;
        fs.n_not_converged = c.n_not_converged;
        fs.n_degenerate = c.n_degenerate;
        fs.max_col_sweeps = c.max_col_sweeps;
        fs.max_col_outer = c.outer_max;
        fs.block_columns = c.block_cols;
        fs.rows_moved = (int64_t)c.rows_moved;
        fs.lambda0 = f.lambda0;
        fill_diagnostics(c, &fs);
        if (fs.diagnostics) {
            agg.diagnostics = 1;
            agg.kkt_viol = std::max(agg.kkt_viol, fs.kkt_viol);
            agg.dual_gap = std::max(agg.dual_gap, fs.dual_gap);
            agg.err_est = std::max(agg.err_est, fs.err_est);
        }
        if (s < 0 && (worst >= 0 || s < worst)) worst = s;
        else if (s > 0 && worst == SPMESL_OK) worst = s;
        agg.outer_iters = std::max(agg.outer_iters, c.outer_max);
        agg.inner_sweeps += (int64_t)c.total_sweeps;
        agg.moves += (int64_t)c.moves;
        agg.active_sweeps += (int64_t)c.act_sweeps;
        agg.active_moves += (int64_t)c.act_moves;
        agg.nnz_B += (int64_t)c.nnz;
        agg.n_not_converged += c.n_not_converged;
        agg.n_degenerate += c.n_degenerate;
        agg.max_col_sweeps = std::max(agg.max_col_sweeps, c.max_col_sweeps);
        agg.max_col_outer = std::max(agg.max_col_outer, c.outer_max);
        agg.block_columns += c.block_cols;
        agg.rows_moved += (int64_t)c.rows_moved;
    }
    agg.status = worst;
    if (b->ev_recorded) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, b->ev[0], b->ev[1]) == cudaSuccess) agg.ms_cd = ms;
    }
    if (stats) *stats = agg;
    return worst;
}

spmesl_status spmesl_batch_fit_stats(const spmesl_batch* b, int i, spmesl_stats* stats) {
    if (!b || !stats || i < 0 || i >= b->count) return SPMESL_EINVAL;
    if ((int)b->fit_stats.size() != b->count) return SPMESL_ENOTFOUND;   // no result read yet
    *stats = b->fit_stats[i];
    return SPMESL_OK;
}

spmesl_status spmesl_batch_tune(spmesl_batch* b, void* workspace, size_t ws_bytes, void* stream,
                                int* best_warps) {
    if (!b) return SPMESL_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int saved_graph = b->use_graph;
    b->use_graph = 0;
    static const int cand[] = {2, 4, 6, 8, 12, 16};
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        return SPMESL_ECUDA;
    float best = 1e30f;
    int bestW = auto_warps(b);
    for (int W : cand) {
        // with the lazy gradient W shapes only the lazy launch, capped at LAZY_MAX_WARPS
        if (b->gradient != SPMESL_GRADIENT_EAGER && W > LAZY_MAX_WARPS) continue;
        b->warps_per_block = W;
        float tot = 0.f;
        bool ok = true;
        for (int rep = 0; rep < 3 && ok; ++rep) {
            cudaEventRecord(e0, st);
            ok = spmesl_batch_run(b, workspace, ws_bytes, stream) == SPMESL_OK;
            cudaEventRecord(e1, st);
            if (ok && cudaEventSynchronize(e1) == cudaSuccess) {
                float ms = 0.f;
                cudaEventElapsedTime(&ms, e0, e1);
                if (rep > 0) tot += ms;           // first run warms up
            } else {
                ok = false;
            }
        }
        if (ok && tot < best) {
            best = tot;
            bestW = W;
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->warps_per_block = bestW;
    b->use_graph = saved_graph;
    if (best_warps) *best_warps = bestW;
    return best < 1e29f ? SPMESL_OK : SPMESL_ECUDA;
}

spmesl_status spmesl_batch_tune_cached(spmesl_batch* b, void* workspace, size_t ws_bytes,
                                       void* stream, const char* cache_path,
                                       spmesl_tune_choice* out) {
    if (!b || !workspace) return SPMESL_EINVAL;
    double nsum = 0.0;
    int nx = 0;
    for (const FitPlan& f : b->plan)
        if (f.X) {
            nsum += f.n;
            ++nx;
        }
    char key[256];
    if (spmesl_tune_key(b->precision, b->standardize, num_sms(), b->count, b->max_p,
                        nx ? nsum / nx : 1.0, key, sizeof(key)) < 0)
        return SPMESL_EINVAL;
    spmesl_tune_choice c{};
    if (cache_path && spmesl_tune_cache_lookup(cache_path, key, &c) == SPMESL_OK) {
        b->warps_per_block = c.warps_per_block;
        b->handover = c.handover;
        b->heavy_min_p = c.heavy_min_p;
        b->heavy_heat = c.heavy_heat;
        if (out) *out = c;
        return SPMESL_OK;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int saved_graph = b->use_graph;
    b->use_graph = 0;
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess)
        return SPMESL_ECUDA;
    const bool lazy = b->gradient != SPMESL_GRADIENT_EAGER;
    const bool route = b->gradient == SPMESL_GRADIENT_AUTO;
    static const int wl[] = {4, 8}, we[] = {2, 4, 8, 16};
    static const int hv[] = {32, 64}, mp[] = {0, 1024, -1};
    const int* ws_ = lazy ? wl : we;
    const int nw = lazy ? 2 : 4, nh = route ? 2 : 1, nm = (route && b->standardize) ? 3 : 1;
    float best = 1e30f;
    spmesl_tune_choice bc{b->warps_per_block, b->handover, b->heavy_min_p, b->heavy_heat, 0.f, 0};
    bool ok = true;
    for (int iw = 0; iw < nw && ok; ++iw)
        for (int ih = 0; ih < nh && ok; ++ih)
            for (int im = 0; im < nm && ok; ++im) {
                b->warps_per_block = ws_[iw];
                if (route) b->handover = hv[ih];
                if (route && b->standardize) b->heavy_min_p = mp[im];
                float tot = 0.f;
                for (int rep = 0; rep < 3 && ok; ++rep) {
                    cudaEventRecord(e0, st);
                    ok = spmesl_batch_run(b, workspace, ws_bytes, stream) == SPMESL_OK;
                    cudaEventRecord(e1, st);
                    if (ok && cudaEventSynchronize(e1) == cudaSuccess) {
                        float ms = 0.f;
                        cudaEventElapsedTime(&ms, e0, e1);
                        if (rep > 0) tot += ms;           // the first run warms up
                    } else {
                        ok = false;
                    }
                }
                if (ok && tot / 2 < best) {
                    best = tot / 2;
                    bc = spmesl_tune_choice{b->warps_per_block, b->handover, b->heavy_min_p,
                                            b->heavy_heat, best, 0};
                }
            }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    b->warps_per_block = bc.warps_per_block;
    b->handover = bc.handover;
    b->heavy_min_p = bc.heavy_min_p;
    b->use_graph = saved_graph;
    if (!ok) return SPMESL_ECUDA;
    if (cache_path && spmesl_tune_cache_store(cache_path, key, &bc) != SPMESL_OK)
        return SPMESL_EINVAL;
    if (out) *out = bc;
    return SPMESL_OK;
}

void spmesl_batch_destroy(spmesl_batch* b) {
    if (!b) return;
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
    if (b->side2) cudaStreamDestroy(b->side2);
    if (b->fork2) cudaEventDestroy(b->fork2);
    if (b->join2) cudaEventDestroy(b->join2);
    if (b->ev[0]) cudaEventDestroy(b->ev[0]);
    if (b->ev[1]) cudaEventDestroy(b->ev[1]);
    if (b->pinned) {
        if (b->pinned_is_pageable) std::free(b->pinned);
        else cudaFreeHost(b->pinned);
    }
    delete b;
}

}  // extern "C"
