#pragma once
// Device building blocks of the coordinate-descent fit, shared by the single-fit
// kernels (cd.cu) and the batched kernels (batch.cu).
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>

#include "common.cuh"

namespace spmesl {

template <typename T>
struct CDArgs {
    const T* SC;
    T* BT;
    T* GT;
    const T* diag;       // S_kk of the working matrix (unstandardised update); with chunk_max
                         // (standardised lazy solves) max_k |S^C_jk|, k != j, instead
    double* sigma;       // working-scale sigma
    int* col_status;
    int* active;
    int* active_next;
    int* flag;
    FitCtrl* ctrl;
    int p, ldp, maxit;
    double lambda0, tol;
    float tolf;          // the smallest float not below tol (see float_at_least)
    int* ovf_list;       // columns handed from the lazy solver to the block solver
    int* ovf_count;
    const int* order;    // queue order of the lazy solver (nullptr: 0..p-1)
    int n_queue;         // columns the lazy solver takes from its queue
    int ovf_supp;        // the lazy solver hands a column over when its support exceeds this
                         // at the start of an active-set phase (ACT_MAX with heavy-column
                         // routing, LAZY_CAP without)
    const float* chunk_max;   // per column j and 128-coordinate chunk c, max_k |S^C_jk| over
                              // the chunk (k != j), written by the standardisation pass; the
                              // first sweep's skip test starts from it (nullptr: scan all)
    unsigned* rows_moved;     // measurement (nullptr: off): bit k of row m is set when
                              // coordinate k moved in the m-th full sweep of any column
    int rows_words;           // 32-bit words per row of that bitmap
    double* hand;             // per column the last sigma step (sigma, F(sigma)) at a hand-over
                              // from the lazy to the block solver (nullptr: the block solver
                              // starts every column afresh); of a batch's solved column the
                              // second is sigma^2, for sqrt_last
    int* nsup;                // per column the entries of its list in row j of BT, -1 when the
                              // row is dense (nullptr: every row is dense)
    double* Theta;            // the column solvers clear row j of it (nullptr: not)
};

// The solved columns' coefficients.  Row j of BT holds b_j as a list when it
// has at most coef_cap(ldp) nonzero coefficients: the values in ascending order
// of their coordinates at the start of the row and the coordinates (int) from
// its middle, their number in nsup[j]; otherwise the row is dense and nsup[j]
// is -1.  A row of Theta is nonzero only where both regressions of the pair
// have a nonzero coefficient (the smaller magnitude of the two is taken), so
// Theta is its diagonal and a few entries per row: the solvers clear row j of
// Theta when they have solved column j (streaming stores under their own
// compute), and theta_column writes the nonzero entries from the lists.
constexpr int COEF_CAP = 1024;
__host__ __device__ constexpr int coef_cap(int ldp) {
    return ldp / 2 < COEF_CAP ? ldp / 2 : COEF_CAP;
}
template <typename T>
__device__ __forceinline__ int* coef_idx(T* row, int ldp) {
    return reinterpret_cast<int*>(row + ldp / 2);
}
template <typename T>
__device__ __forceinline__ const int* coef_idx(const T* row, int ldp) {
    return reinterpret_cast<const int*>(row + ldp / 2);
}

// b_kj (the coefficient of x_k in regression j) from row j of BT.
template <typename T>
__device__ __forceinline__ T coef_of(const T* __restrict__ BT, const int* __restrict__ nsup, int ldp,
                                     int j, int k) {
    const T* __restrict__ row = BT + (size_t)j * ldp;
    const int n = nsup ? nsup[j] : -1;
    if (n < 0) return row[k];
    const int* __restrict__ idx = coef_idx(row, ldp);
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (idx[mid] < k) lo = mid + 1;
        else hi = mid;
    }
    return lo < n && idx[lo] == k ? row[lo] : T(0);
}

// Row j of Theta cleared by `nthr` threads with 16-byte streaming stores (the
// lines are not read again before theta_column, so they leave L2 first).
__device__ __forceinline__ void clear_theta_row(double* __restrict__ Theta, int p, int j, int tid,
                                                int nthr) {
    double* __restrict__ row = Theta + (size_t)j * p;
    const int head = (reinterpret_cast<uintptr_t>(row) & 15) ? 1 : 0;
    const int nv = (p - head) / 2;
    double2* __restrict__ v = reinterpret_cast<double2*>(row + head);
    for (int i = tid; i < nv; i += nthr) __stcs(v + i, make_double2(0.0, 0.0));
    if (tid == 0) {
        if (head) row[0] = 0.0;
        if (head + 2 * nv < p) row[p - 1] = 0.0;
    }
}

// Full sweeps per column whose moved coordinates are recorded in the bitmap.
constexpr int ROWS_SWEEPS = 64;

// ctrl->rows_moved += the set bits of bits[0, nwords) (grid-stride).
__device__ __forceinline__ void count_rows_moved(const unsigned* __restrict__ bits, size_t nwords,
                                                 FitCtrl* ctrl, size_t tid, size_t nthr) {
    unsigned long long c = 0;
    for (size_t i = tid; i < nwords; i += nthr) c += __popc(bits[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(FULL_MASK, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(&ctrl->rows_moved, c);
}

// Record that coordinate k moved in full sweep m (one thread calls it).
template <typename T>
__device__ __forceinline__ void note_row_moved(const CDArgs<T>& a, int m, int k) {
    if (a.rows_moved && m >= 0 && m < ROWS_SWEEPS)
        atomicOr(a.rows_moved + (size_t)m * a.rows_words + (k >> 5), 1u << (k & 31));
}

namespace {
// Order of a coordinate-descent queue: columns by decreasing heat (the count
// of off-diagonal standardised entries above lambda0, from standardize_row;
// counting sort, one block), so the longest column solves start first instead
// of in the tail of the launch.  Ties in any order: a column's result does not
// depend on when it runs.  With n_heavy, also the number of columns whose heat
// exceeds heavy_heat (< HEAT_BINS - 1): they lead the order and go to the
// block solver.
constexpr int HEAT_BINS = 64;
__global__ void __launch_bounds__(1024) order_by_heat_kernel(const int* __restrict__ heat, int n,
                                                          int* __restrict__ order,
                                                          int* __restrict__ n_heavy,
                                                          int heavy_heat) {
    __shared__ int bin[HEAT_BINS];
    const int t = threadIdx.x;
    if (t < HEAT_BINS) bin[t] = 0;
    __syncthreads();
    for (int i = t; i < n; i += blockDim.x) atomicAdd(&bin[min(heat[i], HEAT_BINS - 1)], 1);
    __syncthreads();
    if (t == 0) {
        int run = 0;
        for (int h = HEAT_BINS - 1; h >= 0; --h) {
            const int c = bin[h];
            bin[h] = run;
            run += c;
            if (h == heavy_heat + 1 && n_heavy) *n_heavy = run;
        }
    }
    __syncthreads();
    for (int i = t; i < n; i += blockDim.x) order[atomicAdd(&bin[min(heat[i], HEAT_BINS - 1)], 1)] = i;
}
}  // namespace

template <typename T>
__device__ __forceinline__ T soft(T x, T lam) {
    // Soft_lambda(x) = sign(x) (|x| - lambda)_+   (Section 3.1)
    return x > lam ? x - lam : (x < -lam ? x + lam : T(0));
}

// The same for the standardised working matrix, where every operand is finite
// (|S| <= 1; non-finite input ends the fit before its solvers), in fewer
// dependent instructions.  FP32: x minus x clamped to [-lambda, lambda], two
// min/max operations in place of two compares and two selects.  FP64: one
// FP64 addition; the compare is of the magnitudes' bits, since every FP64
// compare, minimum or conversion takes a slot of the FP64 pipe (16 cycles a
// warp on this part).
__device__ __forceinline__ float soft_std(float x, float lam) {
    return x - fminf(fmaxf(x, -lam), lam);
}
__device__ __forceinline__ long long abs_bits(double x) {
    return __double_as_longlong(x) & 0x7fffffffffffffffll;
}
__device__ __forceinline__ double soft_std(double x, double lam) {
    const long long sgn = __double_as_longlong(x) & (long long)0x8000000000000000ull;
    const double y = x - __longlong_as_double(__double_as_longlong(lam) | sgn);
    return abs_bits(x) > __double_as_longlong(lam) ? y : 0.0;
}

// a != b for coefficients (never -0: soft_std gives +0 or a nonzero value).
__device__ __forceinline__ bool differs(float a, float b) { return a != b; }
__device__ __forceinline__ bool differs(double a, double b) {
    return __double_as_longlong(a) != __double_as_longlong(b);
}

// Running max |d| and the change test of the phases' moves, without the FP64 pipe.
__device__ __forceinline__ float max_abs(float m, float d) { return fmaxf(m, fabsf(d)); }
__device__ __forceinline__ double max_abs(double m, double d) {
    const long long a = __double_as_longlong(m), b = abs_bits(d);
    return __longlong_as_double(b > a ? b : a);
}
__device__ __forceinline__ bool is_move(float d) { return d != 0.0f; }
__device__ __forceinline__ bool is_move(double d) { return abs_bits(d) != 0; }

// |x| as a float that is not below it (a bound): for FP64 from the upper word,
// rounded up by one unit of it, so that no FP64 conversion is needed per value.
__device__ __forceinline__ unsigned abs_key(float x) { return __float_as_uint(fabsf(x)); }
__device__ __forceinline__ unsigned abs_key(double x) {
    return (unsigned)(__double_as_longlong(x) >> 32) & 0x7fffffffu;
}
// Keys from here on are infinities and NaN.
template <typename T>
__device__ constexpr unsigned key_nonfinite() { return sizeof(T) == 4 ? 0x7f800000u : 0x7ff00000u; }
// |x| > lam for lam >= 0.
__device__ __forceinline__ bool abs_above(float x, float lam) { return fabsf(x) > lam; }
__device__ __forceinline__ bool abs_above(double x, double lam) {
    return abs_bits(x) > __double_as_longlong(lam);
}
// The value that a key stands for, as a float bound.
template <typename T>
__device__ __forceinline__ float key_bound(unsigned m) {
    if constexpr (sizeof(T) == 4) return __uint_as_float(m);
    else return __double2float_ru(__hiloint2double((int)(m + 1u), 0));
}
// The largest key of the warp (non-negative floats and the upper words of
// non-negative doubles order as unsigned integers).
template <typename T>
__device__ __forceinline__ float warp_max_key(unsigned key) {
    return key_bound<T>(__reduce_max_sync(0xffffffffu, key));
}

// The smallest float f >= x.  For a float m, m < x exactly when m < f, so a
// stop test of a float iterate against the FP64 tolerance needs no FP64
// arithmetic per test.
inline float float_at_least(double x) {
    float f = (float)x;
    if ((double)f < x) f = nextafterf(f, INFINITY);
    return f;
}

// md < tol for an iterate of the working precision T (float: against the
// float threshold tf of float_at_least(tol); double: directly).
template <typename T>
__device__ __forceinline__ bool below_tol(T md, double tol, float tf) {
    if constexpr (sizeof(T) == 4) return md < tf;
    else return (double)md < tol;
}

template <typename T>
__device__ __forceinline__ T warp_max(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(FULL_MASK, v, o));
    return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL_MASK, v, o);
    return v;
}

// (double)x without the FP64 pipe, where a conversion takes as long as an
// addition: the exponent rebased and the fraction moved, by integer
// instructions.  Denormal FP32 values, infinities and NaN take the conversion.
__device__ __forceinline__ double exact_double(float x) {
    const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u && m != 0u) return (double)x;
    const unsigned hi = (u & 0x80000000u) | (m != 0u ? (m >> 3) + 0x38000000u : 0u);
    return __hiloint2double((int)hi, (int)(u << 29));
}
__device__ __forceinline__ double exact_double(double x) { return x; }

// Ordered bits of a non-negative double (for atomicMax).
__device__ __forceinline__ unsigned long long dbits(double x) {
    return (unsigned long long)__double_as_longlong(x);
}

// dst[0..ldp) = src[0..ldp) with 16-byte vectors (one warp).
template <typename T>
__device__ __forceinline__ void warp_copy(T* __restrict__ dst, const T* __restrict__ src, int ldp) {
    using V = typename Vec16<T>::type;
    constexpr int N = Vec16<T>::N;
    const int lane = threadIdx.x & 31;
    for (int l = lane * N; l < ldp; l += 32 * N)
        *reinterpret_cast<V*>(dst + l) = *reinterpret_cast<const V*>(src + l);
}

template <typename T>
__device__ __forceinline__ void warp_zero(T* __restrict__ dst, int ldp) {
    using V = typename Vec16<T>::type;
    constexpr int N = Vec16<T>::N;
    const int lane = threadIdx.x & 31;
    V z;
    if constexpr (N == 4) z = make_float4(0.f, 0.f, 0.f, 0.f);
    else z = make_double2(0.0, 0.0);
    for (int l = lane * N; l < ldp; l += 32 * N) *reinterpret_cast<V*>(dst + l) = z;
}

// g[l] -= srow[l] * delta for l in [0, ldp): the column-j slice of the rank-1
// update G -= S_.k delta_k. (Proposition 2 on the covariance.)
template <typename T>
__device__ __forceinline__ void axpy_row(T* __restrict__ g, const T* __restrict__ srow, T delta,
                                         int ldp) {
    const int lane = threadIdx.x & 31;
    if constexpr (sizeof(T) == 4) {
        for (int l = lane * 4; l < ldp; l += 128) {
            const float4 s = __ldg(reinterpret_cast<const float4*>(srow + l));
            float4 v = *reinterpret_cast<float4*>(g + l);
            v.x = fmaf(-s.x, delta, v.x);
            v.y = fmaf(-s.y, delta, v.y);
            v.z = fmaf(-s.z, delta, v.z);
            v.w = fmaf(-s.w, delta, v.w);
            *reinterpret_cast<float4*>(g + l) = v;
        }
    } else {
        for (int l = lane * 2; l < ldp; l += 64) {
            const double2 s = __ldg(reinterpret_cast<const double2*>(srow + l));
            double2 v = *reinterpret_cast<double2*>(g + l);
            v.x = fma(-s.x, delta, v.x);
            v.y = fma(-s.y, delta, v.y);
            *reinterpret_cast<double2*>(g + l) = v;
        }
    }
}

// One cyclic ascending sweep over k != j for column j (Algorithm 1's inner
// loop, written on g = S_.j - S b).  Returns max |delta b| over the sweep
// (same value in every lane); `moves` counts coordinates that changed.
// Four consecutive elements starting at a 4-aligned index (16-byte or 2 x
// 16-byte shared-memory loads).
template <typename T>
__device__ __forceinline__ void load4(const T* __restrict__ src, T (&v)[4]) {
    if constexpr (sizeof(T) == 4) {
        const float4 q = *reinterpret_cast<const float4*>(src);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        const double2 q0 = *reinterpret_cast<const double2*>(src);
        const double2 q1 = *reinterpret_cast<const double2*>(src + 2);
        v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
    }
}

// Each lane evaluates 4 consecutive coordinates, so one step of the warp
// covers a 128-coordinate chunk; the first coordinate whose update changes b
// is applied and the scan resumes right after it within the chunk.
constexpr int SCAN_V = 4;
constexpr int CHUNK = 32 * SCAN_V;

// Per-chunk summary kept between sweeps for the skip test (standardised
// working matrix only): after the chunk was last scanned, the largest |g_k|
// over its coordinates with b_k = 0, how many of its b_k were nonzero, and
// the running sum of |delta| and move count at that moment.
struct ChunkInfo {
    float maxabs;
    float dsum_at;
    unsigned moves_at;
    int nsupp;
};

// Scan state of one column solve (warp-uniform).
struct ColScan {
    ChunkInfo* ci;
    float dsum;          // running sum of the size of every change of b_j so far: one
                         // move's |delta|, or an active-set phase's net change; in the lazy
                         // solver each |delta_m| times max_k |S_mk|
    unsigned nmoves;     // number of those changes
    float bl1;           // lazy solver: an upper bound of ||b_j||_1 so far (0 elsewhere)
};

// A chunk with no support can be skipped when no coordinate in it can reach
// the threshold: each move delta_m at row m changes g_k by -S_km delta_m with
// |S_km| <= 1 (standardised), so |g_k| <= maxabs + sum|delta| since the chunk
// was scanned (and a change of several coefficients at once moves g_k by at
// most its l1 size).  The lazy solver counts each |delta_m| times the largest
// off-diagonal |S_mk| of row m (an Erdos-Renyi column at p = 2000 forms 6.2
// slices instead of 10.1, one of an AR(1) network at p = 1000 13.1 instead of
// 16.8).  It forms g_k afresh from S rows at every
// scan: each of the two computations (then and now) is off by at most
// 384 * 2^-24 (1 + ||b||_1) (up to 256 support rows and 128 moves in a
// chunk, |S| <= 1), the last term below with bl1 bounding ||b||_1 then and now.  The margins cover FP32 rounding of the standardised S
// (|S_km| <= 1 + 2^-22), of every g update (half an ulp of a value below
// lambda) and of the running sum (each of the dm additions since the scan is
// off by at most 2^-24 of the sum, which only grows); after 4096 moves the
// chunk is always rescanned.  A skipped coordinate therefore has
// |g_k| < lambda and b_k = 0, so it would not have moved: the sweep is the
// same as a full scan.  With `frozen` (a sweep that leaves the support's
// values as they are, see solve_column_lazy) a chunk holding support may be
// skipped too: maxabs covers the chunk's coordinates that were zero when it
// was scanned, and a coordinate that has left the support since then marks
// its chunk for a rescan (maxabs = infinity).
__device__ __forceinline__ bool chunk_skippable(const ChunkInfo& c, const ColScan& cs, float lam,
                                                bool frozen = false) {
    const unsigned dm = cs.nmoves - c.moves_at;
    if ((c.nsupp != 0 && !frozen) || dm > 4096u) return false;
    const float dd = cs.dsum - c.dsum_at;
    const float bound = c.maxabs + dd * (1.0f + 0x1p-10f) + cs.dsum * (float)(dm + 2u) * 0x1p-23f +
                        (float)dm * lam * 0x1p-20f + (1.0f + cs.bl1 + dd) * 0x1p-14f;
    return bound < lam;
}

// An upper bound of the warp's sum of |x| (one hardware reduction): each |x|
// rounded up to a multiple of 2^-20; infinite when the sum reaches 64.
__device__ __forceinline__ float warp_l1_bound(float x) {
    const unsigned q = __float2uint_ru(fminf(fabsf(x), 64.0f) * 0x1p20f);
    const unsigned t = __reduce_add_sync(FULL_MASK, q);
    return t >= (1u << 26) ? INFINITY : __uint2float_ru(t) * 0x1p-20f;
}

template <typename T, bool STD>
__device__ T sweep_column(int j, T* __restrict__ g, T* __restrict__ b, const CDArgs<T>& a, T lam,
                          unsigned long long& moves, ColScan& cs, int sweep_idx = -1) {
    const int lane = threadIdx.x & 31;
    const int p = a.p;
    const int ldp = a.ldp;
    T maxd = T(0);
    for (int cb = 0, ci = 0; cb < p; cb += CHUNK, ++ci) {
        if constexpr (STD) {
            if (chunk_skippable(cs.ci[ci], cs, (float)lam)) continue;
        }
        const int k0 = cb + lane * SCAN_V;
        int cursor = cb;
        for (;;) {
            T gv[SCAN_V], bv[SCAN_V], nbv[SCAN_V];
            if (k0 < ldp) {                   // ldp is a multiple of 32: the whole quad is in range
                load4<T>(g + k0, gv);
                load4<T>(b + k0, bv);
            } else {
#pragma unroll
                for (int t = 0; t < SCAN_V; ++t) gv[t] = bv[t] = T(0);
            }
            unsigned mvmask = 0u;
#pragma unroll
            for (int t = 0; t < SCAN_V; ++t) {
                const int k = k0 + t;
                nbv[t] = bv[t];
                if (k >= cursor && k < p && k != j) {
                    T nb;
                    if constexpr (STD) {
                        nb = soft<T>(gv[t] + bv[t], lam);                  // S_kk = 1
                    } else {
                        const T skk = a.diag[k];
                        nb = soft<T>(gv[t] + skk * bv[t], lam) / skk;      // Soft(c, lambda)/S_kk
                    }
                    nbv[t] = nb;
                    if (nb != bv[t]) mvmask |= 1u << t;
                }
            }
            const unsigned bal = __ballot_sync(FULL_MASK, mvmask != 0u);
            if (bal == 0u) break;
            const int f = __ffs(bal) - 1;
            const int tf = __ffs(__shfl_sync(FULL_MASK, mvmask, f)) - 1;
            T nb_sel = nbv[0], b_sel = bv[0];
#pragma unroll
            for (int t = 1; t < SCAN_V; ++t)
                if (t == tf) { nb_sel = nbv[t]; b_sel = bv[t]; }
            const T nbs = __shfl_sync(FULL_MASK, nb_sel, f);
            const T delta = nbs - __shfl_sync(FULL_MASK, b_sel, f);
            const int ks = cb + f * SCAN_V + tf;
            if (lane == 0) {
                b[ks] = nbs;
                note_row_moved(a, sweep_idx, ks);
            }
            maxd = fmax(maxd, fabs(delta));
            ++moves;
            cs.dsum += fabsf((float)delta);
            ++cs.nmoves;
            axpy_row<T>(g, a.SC + (size_t)ks * ldp, delta, ldp);
            __syncwarp();
            cursor = ks + 1;
            if (cursor >= cb + CHUNK) break;
        }
        if constexpr (STD) {
            // summary of the chunk as it leaves the scan
            float mx = 0.f;
            int ns = 0;
            if (k0 < ldp) {
                T gv[SCAN_V], bv[SCAN_V];
                load4<T>(g + k0, gv);
                load4<T>(b + k0, bv);
#pragma unroll
                for (int t = 0; t < SCAN_V; ++t) {
                    const int k = k0 + t;
                    if (k < p && k != j) {
                        if (bv[t] != T(0)) ++ns;
                        else mx = fmaxf(mx, fabsf((float)gv[t]));
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                mx = fmaxf(mx, __shfl_xor_sync(FULL_MASK, mx, o));
                ns += __shfl_xor_sync(FULL_MASK, ns, o);
            }
            if (lane == 0) cs.ci[ci] = ChunkInfo{mx, cs.dsum, cs.nmoves, ns};
            __syncwarp();
        }
    }
    return maxd;
}

// Mark every chunk "must scan" (maxabs = infinity fails every skip test).
__device__ __forceinline__ void reset_chunks(ColScan& cs, int ldp) {
    const int nc = (ldp + CHUNK - 1) / CHUNK;
#pragma unroll 1
    for (int c = threadIdx.x & 31; c < nc; c += 32) cs.ci[c] = ChunkInfo{INFINITY, 0.f, 0u, 1};
    cs.dsum = 0.f;
    cs.nmoves = 0u;
    cs.bl1 = 0.f;
}

// Per-warp scratch for the support list used by the sigma update.
constexpr int SUPP_CAP = 128;

// Shared memory of one warp: g_j and b_j (ldp elements each), the support
// list and the chunk summaries.
__host__ __device__ constexpr int num_chunks(int ldp) { return (ldp + CHUNK - 1) / CHUNK; }

template <typename T>
__host__ __device__ constexpr size_t warp_smem_bytes(int ldp) {
    return 2 * (size_t)ldp * sizeof(T) + SUPP_CAP * sizeof(int) +
           (size_t)num_chunks(ldp) * sizeof(ChunkInfo);
}

// sigma_j^2 = S_jj - 2 b'S_.j + b'S b in FP64 over the support of b
// (Eq. (14) written on S).  Same value in every lane.
template <typename T>
__device__ double residual_quadratic_form(int j, const T* __restrict__ b, const CDArgs<T>& a,
                                          int* __restrict__ list) {
    const int lane = threadIdx.x & 31;
    const int p = a.p;
    // support of b in ascending order
    int ns = 0;
    for (int c0 = 0; c0 < p; c0 += 32) {
        const int k = c0 + lane;
        const bool nz = k < p && b[k] != T(0);
        const unsigned bal = __ballot_sync(FULL_MASK, nz);
        if (nz) {
            const int pos = ns + __popc(bal & ((1u << lane) - 1u));
            if (pos < SUPP_CAP) list[pos] = k;
        }
        ns += __popc(bal);
    }
    __syncwarp();
    double lin = 0.0, quad = 0.0;
    if (ns <= SUPP_CAP) {
        for (int t = lane; t < ns; t += 32) {
            const int k = list[t];
            lin = fma((double)b[k], (double)a.SC[(size_t)k * a.ldp + j], lin);
        }
        // rows of the support in turn, lanes over its columns (FP64 products)
        for (int u = 0; u < ns; ++u) {
            const int k = list[u];
            const T* __restrict__ row = a.SC + (size_t)k * a.ldp;
            double part = 0.0;
            for (int v = lane; v < ns; v += 32) {
                const int l = list[v];
                part = fma((double)b[l], (double)row[l], part);
            }
            quad = fma((double)b[k], part, quad);
        }
        lin = warp_sum(lin);
        quad = warp_sum(quad);
        __syncwarp();
        return (double)a.SC[(size_t)j * a.ldp + j] - 2.0 * lin + quad;
    }
    // large support: row-wise accumulation without the list
    for (int c0 = 0; c0 < p; c0 += 32) {
        const int k = c0 + lane;
        const T bk = (k < p) ? b[k] : T(0);
        unsigned bal = __ballot_sync(FULL_MASK, bk != T(0));
        while (bal) {
            const int f = __ffs(bal) - 1;
            bal &= bal - 1;
            const int kk = c0 + f;
            const double bkk = (double)__shfl_sync(FULL_MASK, bk, f);
            const T* srow = a.SC + (size_t)kk * a.ldp;
            double part = 0.0;
            for (int l = lane; l < p; l += 32) {
                const T bl = b[l];
                if (bl != T(0)) part += (double)bl * (double)srow[l];
            }
            quad += bkk * part;
            if (lane == 0) lin += bkk * (double)srow[j];
        }
    }
    lin = warp_sum(lin);
    quad = warp_sum(quad);
    return (double)a.SC[(size_t)j * a.ldp + j] - 2.0 * lin + quad;
}

// Row r of S^C = C S C into SC (zero padding up to ldp), optionally copied
// into GT.  FP32 data is scaled in FP32 by the scales
// rounded once to FP32 (csf); FP64 data in FP64.  One warp takes one
// 128-coordinate chunk of the row at a time (threads tid, tid + nthr, ...;
// nthr a multiple of 32).  Optional outputs: heat, this thread's count of
// off-diagonal |SC_rc| > heat_lam; cmax, per chunk c of the row the largest
// off-diagonal |SC_rk| (row r of a p x num_chunks(ldp) table; S^C is
// symmetric, so it is also column r's first-sweep gradient bound); with it,
// *rowmax takes the largest of the warp's chunks and diag is left to the
// caller (FP64: the bounds of abs_key).  Returns true if a non-finite entry was
// seen.  Of FP64 data only the two products go to the FP64 pipe, which
// otherwise bounds the pass (tests, maximum and conversion are 16 cycles a warp's
// instruction each): 50 fits of p = 500 took 127 us
// with them, 94 without.
constexpr int STD_U = 4;
template <typename T>
__device__ __forceinline__ bool standardize_row(const T* __restrict__ S, int p, int ldp, int r,
                                                const double* __restrict__ cs,
                                                const float* __restrict__ csf,
                                                T* __restrict__ SC, T* __restrict__ GT,
                                                T* __restrict__ diag, int tid,
                                                int nthr, T heat_lam = T(0), int* heat = nullptr,
                                                float* __restrict__ cmax = nullptr,
                                                float* rowmax = nullptr) {
    unsigned seen = 0u;                       // largest key of S's entries (a test of each
                                              // FP64 entry would go to the FP64 pipe)
    const int lane = tid & 31;
    const T cr = sizeof(T) == 4 ? (T)csf[r] : (T)cs[r];
    const T* __restrict__ srow = S + (size_t)r * p;
    T* __restrict__ out = SC + (size_t)r * ldp;
    T* __restrict__ grow = GT ? GT + (size_t)r * ldp : nullptr;
    const int nch = num_chunks(ldp);
    const int wstep = nthr >> 5;
    // 16-byte accesses when the rows of S are 16-byte aligned (same arithmetic)
    const bool vec = sizeof(T) == 4 && (p & 3) == 0 && (reinterpret_cast<uintptr_t>(S) & 15) == 0;
    // STD_U chunks per pass: their S values are loaded first, so a warp has
    // STD_U loads in flight instead of one
    for (int chb = tid >> 5; chb < nch; chb += STD_U * wstep) {
        T sv[STD_U][4];
#pragma unroll
        for (int u = 0; u < STD_U; ++u) {
            const int ch = chb + u * wstep;
            const int c0 = ch * CHUNK;
            bool done = false;
            if constexpr (sizeof(T) == 4) {
                if (vec) {                            // lane: coordinates c0 + 4 lane + t
                    const int c = c0 + 4 * lane;
                    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (ch < nch && c < p) q = *reinterpret_cast<const float4*>(srow + c);
                    sv[u][0] = q.x; sv[u][1] = q.y; sv[u][2] = q.z; sv[u][3] = q.w;
                    done = true;
                }
            }
            if (!done) {                              // lane: coordinates c0 + lane + 32 t
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = c0 + lane + 32 * t;
                    sv[u][t] = (ch < nch && c < p) ? srow[c] : T(0);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < STD_U; ++u) {
            const int ch = chb + u * wstep;
            if (ch >= nch) break;                     // warp-uniform
            const int c0 = ch * CHUNK;
            unsigned mx = 0u;                         // largest key (abs_key)
            T v[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int c = vec ? c0 + 4 * lane + t : c0 + lane + 32 * t;
                v[t] = T(0);
                if (c < p) {
                    seen = max(seen, abs_key(sv[u][t]));
                    const T cc = sizeof(T) == 4 ? (T)csf[c] : (T)cs[c];
                    v[t] = sv[u][t] * cr * cc;
                    if (c == r) {
                        if (!cmax) diag[r] = v[t];
                    } else {
                        mx = max(mx, abs_key(v[t]));
                        if (heat && abs_above(v[t], heat_lam)) ++*heat;
                    }
                }
            }
            if (vec) {                                // ldp % 4 == 0: the quad is inside the row
                const int c = c0 + 4 * lane;
                if (c < ldp) {
                    const float4 q = make_float4((float)v[0], (float)v[1], (float)v[2], (float)v[3]);
                    *reinterpret_cast<float4*>(out + c) = q;
                    if (grow) *reinterpret_cast<float4*>(grow + c) = q;
                }
            } else {
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int c = c0 + lane + 32 * t;
                    if (c < ldp) {
                        out[c] = v[t];
                        if (grow) grow[c] = v[t];
                    }
                }
            }
            if (cmax) {
                // (a NaN ends the fit)
                const float top = warp_max_key<T>(mx);
                if (lane == 0) cmax[(size_t)r * nch + ch] = top;
                *rowmax = fmaxf(*rowmax, top);
            }
        }
    }
    return seen >= key_nonfinite<T>();
}

// Per-warp counters of the column solves, flushed into a fit's FitCtrl.
struct ColCounters {
    unsigned long long sweeps = 0, moves = 0;        // full sweeps and their moves
    unsigned long long act_sweeps = 0, act_moves = 0;   // active-set phase
    int outer_max = 0, n_nc = 0, n_deg = 0, max_sw = 0;
    int blk = 0;                                      // columns solved by the block solver
};

__device__ __forceinline__ void flush_counters(FitCtrl* ctrl, ColCounters& c) {
    if ((threadIdx.x & 31) == 0) {
        if (c.sweeps) atomicAdd(&ctrl->total_sweeps, c.sweeps);
        if (c.moves) atomicAdd(&ctrl->moves, c.moves);
        if (c.act_sweeps) atomicAdd(&ctrl->act_sweeps, c.act_sweeps);
        if (c.act_moves) atomicAdd(&ctrl->act_moves, c.act_moves);
        atomicMax(&ctrl->outer_max, c.outer_max);
        atomicMax(&ctrl->max_col_sweeps, c.max_sw);
        if (c.n_nc) atomicAdd(&ctrl->n_not_converged, c.n_nc);
        if (c.n_deg) atomicAdd(&ctrl->n_degenerate, c.n_deg);
    }
    c = ColCounters();
}

// The sigma step of the per-column solvers.  Algorithm 1 iterates the fixed
// point sigma <- F(sigma) = Q(b(sigma lambda0))^1/2 (Eq. (14)), which
// converges linearly.  From the second step on the solvers take the secant
// step on g(s) = F(s) - s through the last two points (s0, F(s0)),
// (s1, F(s1)), kept only when it is positive and within four plain steps of
// [min(s1, F(s1)), max(s1, F(s1))]; otherwise the plain step F(s1).  The stop
// test |F(sigma) - sigma| < tol and the returned pair (b(sigma), F(sigma)) are
// Algorithm 1's, so the fit ends at the same fixed point within tol; about
// 40 % fewer sigma steps reach it.  Any accepted step is a valid next sigma,
// so only the differences are taken in FP64 and the step itself (relative to
// s1) is formed and safeguarded in FP32: FP64 arithmetic is scarce on this
// part and every column takes this step a few times.
// g0 and g1 are (float)(F(s0) - s0) and (float)(f1 - s1).
__device__ __forceinline__ double sigma_step(double s0, float g0, double s1, double f1, float g1) {
    const float ds = (float)(s1 - s0);
    const float den = g1 - g0;
    if (den == 0.0f) return f1;
    const float step = -g1 * (ds / den);                  // candidate - s1
    const float w = 4.0f * fabsf(g1);
    const float lo = fminf(0.0f, g1) - w, hi = fmaxf(0.0f, g1) + w;
    const double cand = s1 + exact_double(step);
    // cand > 0, on the bits
    return (__double_as_longlong(cand) > 0 && step >= lo && step <= hi) ? cand : f1;
}

// |d| < tol (tol > 0) on the bits of d.
__device__ __forceinline__ bool below(double d, double tol) {
    return abs_bits(d) < __double_as_longlong(tol);
}

// False only where q > 1e-12 sjj (sjj > 0) holds: decided on the upper words.  True for
// q < 2^-38 sjj, negative, denormal, infinite or NaN (as on a matrix that is not
// positive semidefinite), which the exact test then decides.
__device__ __forceinline__ bool may_be_floored(double q, double sjj) {
    const int low = max(__double2hiint(sjj) - (39 << 20), 1 << 20) + 1;
    return (unsigned)(__double2hiint(q) - low) >= (unsigned)(0x7ff00000 - low);
}

// sqrt(q) for q > 0 in FP64 by one step of Newton's (Heron's) iteration
// y <- y + (q - y^2) / (2 y) from the FP32 root, with the FP32 reciprocal: the
// FP32 root's relative error of 2^-24 becomes 2^-47 (its square, and the reciprocal's error
// times it), with three instructions on the FP64 pipe.  Outside the FP32 range, sqrt.
static __device__ __noinline__ double sqrt_far(double q) { return sqrt(q); }
__device__ __forceinline__ bool root_in_range(float yf) { return yf > 1e-18f && yf < 1e18f; }
__device__ __forceinline__ double sqrt_heron(double q) {
    const float yf = sqrtf((float)q);
    if (!root_in_range(yf)) return sqrt_far(q);
    const double y0 = exact_double(yf);
    return fma(fma(-y0, y0, q), exact_double(0.5f / yf), y0);
}
// One more step from y = sqrt_heron(q), for a sigma that is returned: within one FP64 unit
// of the root.  A batch takes it with a lane per column after the solvers (the FP64 pipe
// takes as long for one lane as for a warp: a step in each column's solver took 256 mixed
// fits from 1955 to 1993 us); single fits, whose warps leave that pipe idle, in the solver.
__device__ __forceinline__ double sqrt_last(double q, double y) {
    const float yf = (float)y;
    return root_in_range(yf) ? fma(fma(-y, y, q), exact_double(0.5f / yf), y) : y;
}

// Algorithm 1 for response column j, by one warp: warm start from b = 0,
// sigma = 1; lasso sweeps at lambda = sigma * lambda0 until
// max |delta b| < tol; sigma from Eq. (14) in FP64; repeat until sigma moves
// by less than tol.  Writes b_j (row j of BT), sigma_j and the column status.
template <typename T, bool STD>
__device__ void solve_column(int j, T* __restrict__ g, T* __restrict__ b, int* __restrict__ list,
                             const CDArgs<T>& a, ColCounters& cnt) {
    const int lane = threadIdx.x & 31;
    warp_copy<T>(g, a.SC + (size_t)j * a.ldp, a.ldp);   // g = S_.j  (b = 0)
    warp_zero<T>(b, a.ldp);
    ColScan cs{reinterpret_cast<ChunkInfo*>(list + SUPP_CAP), 0.f, 0u};
    reset_chunks(cs, a.ldp);
    __syncwarp();

    double sigma = 1.0;                                  // sigma^(0) = 1
    double s_prev = 0.0, f_prev = 0.0;                   // last (sigma, F(sigma))
    bool have_prev = false;
    const unsigned long long sweeps0 = cnt.sweeps;
    const double floor2 = 1e-12 * (double)a.SC[(size_t)j * a.ldp + j];
    int status = COL_OK;
    int r;
    for (r = 0; r < a.maxit; ++r) {
        const T lam = (T)(sigma * a.lambda0);
        bool inner_ok = false;
        for (int m = 0; m < a.maxit; ++m) {
            const T md = sweep_column<T, STD>(j, g, b, a, lam, cnt.moves, cs,
                                              (int)(cnt.sweeps - sweeps0));
            ++cnt.sweeps;
            if ((double)md < a.tol) {
                inner_ok = true;
                break;
            }
        }
        if (!inner_ok) status |= COL_NOT_CONVERGED;
        double q = residual_quadratic_form<T>(j, b, a, list);
        if (q <= floor2) {
            q = floor2;
            status |= COL_DEGENERATE;
        }
        const double sn = sqrt_heron(q);
        if (fabs(sn - sigma) < a.tol) {
            sigma = sqrt_last(q, sn);
            break;
        }
        double nxt = r + 1 < a.maxit ? sn : sqrt_last(q, sn);
        if (have_prev && r + 1 < a.maxit && !(status & COL_DEGENERATE))
            nxt = sigma_step(s_prev, (float)(f_prev - s_prev), sigma, sn, (float)(sn - sigma));
        s_prev = sigma;
        f_prev = sn;
        have_prev = true;
        sigma = nxt;
    }
    if (r == a.maxit) {
        r = a.maxit - 1;
        status |= COL_NOT_CONVERGED;
    }
    warp_copy<T>(a.BT + (size_t)j * a.ldp, b, a.ldp);
    if (lane == 0) {
        a.sigma[j] = sigma;
        a.col_status[j] = status;
    }
    cnt.outer_max = max(cnt.outer_max, r + 1);
    cnt.max_sw = max(cnt.max_sw, (int)(cnt.sweeps - sweeps0));
    cnt.n_nc += (status & COL_NOT_CONVERGED) != 0;
    cnt.n_deg += (status & COL_DEGENERATE) != 0;
    __syncwarp();
}

// ===========================================================================
// Lazy-gradient column solver.
//
// Algorithm 1 in ascending cyclic order, with an active-set phase before each
// certifying sweep (see solve_column_lazy), and the gradient g = S_.j - S b
// never stored.  The warp keeps only the
// support of b_j, sorted by coordinate, in shared memory.  Each 128-coordinate
// chunk forms its slice of g from coalesced 16-byte reads of row j and of the
// rows of the support (S symmetric), so the chunk's reads are independent and
// cost one round trip.  When a coordinate moves, the rank-1 update
// g -= S_.k delta is applied at once to the rest of the chunk and reaches
// every later chunk when that chunk forms its slice from the updated support.
// This is the covariance form of c = S_kj - sum_{l != k} S_kl b_l.  With about
// 7 KB of shared memory per column instead of two p-vectors, many more columns
// stay resident per SM.
// If the support outgrows the phase or the list, the column is handed to the
// block solver (solve_column_block) through a queue.
// Many warps run this code at different points of it, and its size is what they
// wait for most after S: the 256-fit batch went from 2.55 to 2.19 ms when its
// cold loops were no longer unrolled, the hand-over was written once and the
// integer divisions left it, and to 2.08 ms without the FP64 square root and the
// tolerance's rounding.  Keep cold loops at "unroll 1".
// ===========================================================================
constexpr int LAZY_CAP = 256;

// Supports up to ACT_MAX coordinates get the active-set phase (one
// coordinate per lane, the support's block of S in shared memory).
constexpr int ACT_MAX = 32;

template <typename T>
struct Support {
    int* idx;      // sorted coordinates with b != 0
    T* val;        // their b values
    int n;         // warp-uniform count
};

// The support's entries of S kept in a lazy-solver warp's shared memory, for
// the support `list` (n coordinates; n = -1: none yet): the block S_AA (column k
// at saa + k ACT_MAX), S_jA and S_Aj (the standardised S is rounded by rows and
// then columns, so the two differ in their last bits), and the links and
// coefficients of the FP32 phase.
template <typename T>
struct SupportBlock {
    T* saa;
    T* row;            // S_{j A_m}
    T* col;            // S_{A_m j}
    float* top;        // max_k |S_{A_m k}|, k != A_m (standardised)
    int* list;
    float2* tb;
    int n;
};

// Shared memory of one lazy-solver warp: the support list, the chunk
// summaries, the last sigma step (sigma, F(sigma)) for the secant step (kept
// out of registers) and S_jj, and the support's block of S.
template <typename T>
__host__ __device__ constexpr size_t lazy_warp_smem_bytes(int ldp) {
    return (size_t)LAZY_CAP * (sizeof(int) + sizeof(T)) + (size_t)num_chunks(ldp) * sizeof(ChunkInfo) +
           4 * sizeof(double) + (size_t)ACT_MAX * (ACT_MAX + 2) * sizeof(T) + 2 * ACT_MAX * sizeof(int) +
           (sizeof(T) == 4 ? ACT_MAX * sizeof(float2) : 0);
}

// Set b_k = v in the sorted support (insert, update or remove).  pos is the
// first index with idx[pos] >= k.  Returns false if an insert would overflow.
template <typename T>
__device__ bool support_set(Support<T>& s, int pos, int k, T v) {
    const int lane = threadIdx.x & 31;
    const bool exists = pos < s.n && s.idx[pos] == k;
    if (exists && v != T(0)) {
        if (lane == 0) s.val[pos] = v;
        __syncwarp();
        return true;
    }
    if (!exists && v == T(0)) return true;
    if (!exists && s.n >= LAZY_CAP) return false;
    const int shift = exists ? -1 : 1;
    const int from = exists ? pos + 1 : pos;        // entries [from, n) move by `shift`
    const int cnt = s.n - from;
    // move in register-sized rounds; the direction keeps every read ahead of its write
#pragma unroll 1
    for (int base = 0; base < cnt; base += 32) {
        const int t = shift > 0 ? cnt - 1 - (base + lane) : base + lane;
        int ix = 0;
        T vv = T(0);
        const bool act = (base + lane) < cnt;
        if (act) {
            ix = s.idx[from + t];
            vv = s.val[from + t];
        }
        __syncwarp();
        if (act) {
            s.idx[from + t + shift] = ix;
            s.val[from + t + shift] = vv;
        }
        __syncwarp();
    }
    if (!exists && lane == 0) {
        s.idx[pos] = k;
        s.val[pos] = v;
    }
    s.n += shift;
    __syncwarp();
    return true;
}

template <typename T>
__device__ __forceinline__ void load4g(const T* __restrict__ src, T (&v)[4]) {
    if constexpr (sizeof(T) == 4) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(src));
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        const double2 q0 = __ldg(reinterpret_cast<const double2*>(src));
        const double2 q1 = __ldg(reinterpret_cast<const double2*>(src + 2));
        v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
    }
}

// Chunks of [from, from + 32) that the sweep must scan, as a bit mask: with
// the standardised matrix, a chunk is skipped when chunk_skippable proves
// that none of its coordinates can move; the test reads only the chunk's
// summary and the column's running sums, so the lanes test 32 chunks at once.
// The mask stays valid until a move changes the running sums.
template <bool STD>
__device__ __forceinline__ unsigned chunks_to_scan(const ColScan& cs, int from, int nch, float lam,
                                                   bool frozen) {
    const int ci = from + (int)(threadIdx.x & 31);
    bool need = ci < nch;
    if constexpr (STD) {
        if (need) need = !chunk_skippable(cs.ci[ci], cs, lam, frozen);
    }
    return __ballot_sync(FULL_MASK, need);
}

// The slices of up to scan_group() chunks at once, for a sweep that holds the support
// (at most 32 coordinates, my = this lane's or -1): forms them as the sweep does,
// writes the summaries of the leading chunks in which no coordinate at zero
// passes lambda (there the sweep moves nothing) and returns their number; the
// next chunk's slice, if there is one, is left in `slice` (zero at coordinate j
// and at the support's, which that sweep does not read).  In a
// certifying sweep that is nearly always all of them, and the chunks' loads
// are in flight together: a slice alone is one or a few dependent round trips
// to L2 (2250 cycles at a mean support of 1.4, p = 2000).
template <typename T>
__host__ __device__ constexpr int scan_group() { return sizeof(T) == 4 ? 2 : 1; }
template <typename T, bool STD, int U, int SCAN_G>
__device__ __forceinline__ int scan_quiet_chunks(int j, const Support<T>& s, int my,
                                                 const CDArgs<T>& a, T lam, ColScan& cs,
                                                 const int (&ci)[SCAN_G], int cnt,
                                                 T (&slice)[SCAN_V]) {
    const int lane = threadIdx.x & 31;
    const int ldp = a.ldp;
    const T* __restrict__ Sj = a.SC + (size_t)j * ldp;
    T acc[SCAN_G][SCAN_V];
#pragma unroll
    for (int g = 0; g < SCAN_G; ++g) {
#pragma unroll
        for (int t = 0; t < SCAN_V; ++t) acc[g][t] = T(0);
        const int k0 = ci[g] * CHUNK + lane * SCAN_V;
        if (g < cnt && k0 < ldp) load4g<T>(Sj + k0, acc[g]);
    }
#pragma unroll U
    for (int e = 0; e < s.n; ++e) {
        const T* __restrict__ row = a.SC + (size_t)s.idx[e] * ldp;
        const T v = s.val[e];
        T r[SCAN_G][SCAN_V];
#pragma unroll
        for (int g = 0; g < SCAN_G; ++g) {
            const int k0 = ci[g] * CHUNK + lane * SCAN_V;
            if (g < cnt && k0 < ldp) load4g<T>(row + k0, r[g]);
        }
#pragma unroll
        for (int g = 0; g < SCAN_G; ++g) {
            const int k0 = ci[g] * CHUNK + lane * SCAN_V;
            if (g < cnt && k0 < ldp)
#pragma unroll
                for (int t = 0; t < SCAN_V; ++t) acc[g][t] = fma(-v, r[g][t], acc[g][t]);
        }
    }
    int quiet = 0;
    bool open = true;
#pragma unroll
    for (int g = 0; g < SCAN_G; ++g) {
        if (g < cnt && open) {
            const int k0 = ci[g] * CHUNK + lane * SCAN_V;
            // coordinate j and the support's are not tested
            unsigned held = __ballot_sync(FULL_MASK, my >= 0 && my / CHUNK == ci[g]);
            const int nsupp = __popc(held);
            int skip = j;
            for (;;) {
                const int d = skip - k0;
#pragma unroll
                for (int t = 0; t < SCAN_V; ++t)
                    if (d == t) acc[g][t] = T(0);
                if (held == 0u) break;
                skip = __shfl_sync(FULL_MASK, my, __ffs(held) - 1);
                held &= held - 1u;
            }
            unsigned key = 0u;
#pragma unroll
            for (int t = 0; t < SCAN_V; ++t) key = max(key, abs_key(acc[g][t]));
            const unsigned top = __reduce_max_sync(FULL_MASK, key);
            // FP64 keys are upper words: equal ones go to the exact test too
            open = sizeof(T) == 4 ? top <= abs_key(lam) : top < abs_key(lam);
            if (open) {
                if constexpr (STD) {
                    if (lane == 0)
                        cs.ci[ci[g]] = ChunkInfo{key_bound<T>(top), cs.dsum, cs.nmoves, nsupp};
                }
                quiet = g + 1;
            } else {
#pragma unroll
                for (int t = 0; t < SCAN_V; ++t) slice[t] = acc[g][t];
            }
        }
    }
    __syncwarp();
    return quiet;
}

// One sweep; returns max |delta b|.  Sets `overflow` and stops early if the
// support list is full.  With `frozen` the coordinates in the support keep
// their values and only the others are updated (a coordinate that enters is
// not revisited in the same sweep).
template <typename T, bool STD, int U, int SCAN_G>
__device__ T sweep_column_lazy(int j, Support<T>& s, const CDArgs<T>& a, T lam,
                               unsigned long long& moves, ColScan& cs, bool& overflow,
                               bool frozen, int sweep_idx) {
    const int lane = threadIdx.x & 31;
    const int p = a.p;
    const int ldp = a.ldp;
    const T* __restrict__ Sj = a.SC + (size_t)j * ldp;
    const int nch = (p + CHUNK - 1) / CHUNK;
    T maxd = T(0);
    int e0 = 0;                                   // first support entry with idx >= cb
    int mbase = 0;
    if constexpr (STD) {
        float l1 = 0.f;
#pragma unroll 1
        for (int e = lane; e < s.n; e += 32) l1 += fabsf((float)s.val[e]);
        cs.bl1 = fmaxf(cs.bl1, warp_l1_bound(l1) * (1.0f + 0x1p-16f));
    }
    unsigned mask = chunks_to_scan<STD>(cs, 0, nch, (float)lam, frozen);
    for (;;) {
        if (mask == 0u) {
            mbase += 32;
            if (mbase >= nch) break;
            mask = chunks_to_scan<STD>(cs, mbase, nch, (float)lam, frozen);
            continue;
        }
        T acc[SCAN_V] = {T(0), T(0), T(0), T(0)};
        const bool grouped = frozen && s.n <= 32;
        if (grouped) {
            const int cnt = min(SCAN_G, __popc(mask));
            int g_ci[SCAN_G];
            unsigned left = mask;
#pragma unroll
            for (int g = 0; g < SCAN_G; ++g) {
                g_ci[g] = mbase + __ffs(left) - 1;
                left &= left - 1u;
            }
            const int quiet = scan_quiet_chunks<T, STD, U, SCAN_G>(j, s, lane < s.n ? s.idx[lane] : -1, a, lam,
                                                           cs, g_ci, cnt, acc);
#pragma unroll
            for (int g = 0; g < SCAN_G; ++g)
                if (g < quiet) mask &= mask - 1u;
            if (quiet == cnt) continue;
        }
        const int ci = mbase + __ffs(mask) - 1;
        mask &= mask - 1u;
        const int cb = ci * CHUNK;
#pragma unroll 1
        while (e0 < s.n && s.idx[e0] < cb) ++e0;
        int e1 = e0;
#pragma unroll 1
        while (e1 < s.n && s.idx[e1] < cb + CHUNK) ++e1;
        const int k0 = cb + lane * SCAN_V;
        const bool in = k0 < ldp;                 // the whole quad is inside the padded row
        // slice of g: S_jk - sum_{l in support} S_lk b_l (four rows in flight;
        // an L1 prefetch of all the support rows first was measured slower)
        if (!grouped) {
            const T* __restrict__ col = a.SC + k0;    // column k0 of S; row l at col + l ldp
            if (in) load4g<T>(Sj + k0, acc);
#pragma unroll 4
            for (int e = 0; e < s.n; ++e) {
                const int l = s.idx[e];
                const T v = s.val[e];
                if (in) {
                    T r[SCAN_V];
                    load4g<T>(col + (size_t)l * ldp, r);
#pragma unroll
                    for (int t = 0; t < SCAN_V; ++t) acc[t] = fma(-v, r[t], acc[t]);
                }
            }
        }
        // current b of this lane's coordinates (support entries of the chunk)
        T bv[SCAN_V] = {T(0), T(0), T(0), T(0)};
#pragma unroll 1
        for (int e = e0; e < e1; ++e) {
            const int t = s.idx[e] - k0;
            if (t >= 0 && t < SCAN_V) {
#pragma unroll
                for (int u = 0; u < SCAN_V; ++u)
                    if (u == t) bv[u] = s.val[e];
            }
        }
        const unsigned nmoves0 = cs.nmoves;
        int cursor = cb;
        for (;;) {
            T nbv[SCAN_V];
            unsigned mvmask = 0u;
#pragma unroll
            for (int t = 0; t < SCAN_V; ++t) {
                const int k = k0 + t;
                nbv[t] = bv[t];
                if (k >= cursor && k < p && k != j && !(frozen && bv[t] != T(0))) {
                    T nb;
                    if constexpr (STD) {
                        nb = soft_std(acc[t] + bv[t], lam);                // S_kk = 1
                    } else {
                        const T skk = a.diag[k];
                        nb = soft<T>(acc[t] + skk * bv[t], lam) / skk;     // Soft(c, lambda)/S_kk
                    }
                    nbv[t] = nb;
                    if (STD ? differs(nb, bv[t]) : nb != bv[t]) mvmask |= 1u << t;
                }
            }
            const unsigned bal = __ballot_sync(FULL_MASK, mvmask != 0u);
            if (bal == 0u) break;
            const int f = __ffs(bal) - 1;
            const int tf = __ffs(__shfl_sync(FULL_MASK, mvmask, f)) - 1;
            T nb_sel = nbv[0], b_sel = bv[0];
#pragma unroll
            for (int t = 1; t < SCAN_V; ++t)
                if (t == tf) { nb_sel = nbv[t]; b_sel = bv[t]; }
            const T nbs = __shfl_sync(FULL_MASK, nb_sel, f);
            const T delta = nbs - __shfl_sync(FULL_MASK, b_sel, f);
            const int ks = cb + f * SCAN_V + tf;
            int pos = e0;
#pragma unroll 1
            while (pos < e1 && s.idx[pos] < ks) ++pos;
            const int n_before = s.n;
            if (!support_set<T>(s, pos, ks, nbs)) {
                overflow = true;
                return maxd;
            }
            e1 += s.n - n_before;
            if (lane == 0) note_row_moved(a, sweep_idx, ks);
            if (lane == f) {
#pragma unroll
                for (int u = 0; u < SCAN_V; ++u)
                    if (u == tf) bv[u] = nbs;
            }
            maxd = fmax(maxd, fabs(delta));
            ++moves;
            if constexpr (STD)
                cs.dsum += fabsf((float)delta) * (float)a.diag[ks] * (1.0f + 0x1p-20f);
            ++cs.nmoves;
            cs.bl1 += fabsf((float)delta) * (1.0f + 0x1p-16f);
            // rank-1 update of the rest of this chunk's slice
            if (in) {
                T r[SCAN_V];
                load4g<T>(a.SC + (size_t)ks * ldp + k0, r);
#pragma unroll
                for (int t = 0; t < SCAN_V; ++t) acc[t] = fma(-delta, r[t], acc[t]);
            }
            cursor = ks + 1;
            if (cursor >= cb + CHUNK) break;
        }
        if constexpr (STD) {
            unsigned key = 0u;
#pragma unroll
            for (int t = 0; t < SCAN_V; ++t) {
                const int k = k0 + t;
                if (k < p && k != j && !differs(bv[t], T(0))) key = max(key, abs_key(acc[t]));
            }
            const float mx = warp_max_key<T>(key);
            if (lane == 0) cs.ci[ci] = ChunkInfo{mx, cs.dsum, cs.nmoves, e1 - e0};
            __syncwarp();
            // moves raised the running sums: test the chunks after this one again
            if (cs.nmoves != nmoves0) {
                mbase = ci + 1;
                if (mbase >= nch) break;
                mask = chunks_to_scan<STD>(cs, mbase, nch, (float)lam, frozen);
            }
        } else {
            __syncwarp();
        }
    }
    return maxd;
}

// The sweeps of an active-set phase by one warp, FP32 on the standardised
// matrix (S_kk = 1), on n <= LD coordinates; column k of S_AA at saa + k LD.
// Lane m holds the gradient of coordinate m (g0) and, for LD = 64, of
// coordinate m + 32 (g1); b is in tb[k].y.  One move after another is a chain,
// and a shuffle of the owner's change would be half of it.  So every lane forms
// every move: coordinate k's gradient before move k-1 is shuffled to all lanes
// while move k-1 is formed, and move k first applies the change of move k-1
// with the one entry tb[k].x = S_{A_k A_k-1} (the owner's own fused
// multiply-add, so the iterates are the same bits).  The links, b and the
// columns are read one move ahead; each lane stores the new b itself, so it
// reads back its own value.  A zero change adds exact zeros.
template <int LD>
__device__ __forceinline__ float2 phase_links(const float* __restrict__ saa, float2* __restrict__ tb,
                                              int n, float b0, float b1) {
    const int lane = threadIdx.x & 31;
    if (lane < n) tb[lane] = make_float2(saa[(lane == 0 ? n - 1 : lane - 1) * LD + lane], b0);
    if (LD > 32 && lane + 32 < n)
        tb[lane + 32] = make_float2(saa[(lane + 31) * LD + lane + 32], b1);
    __syncwarp();
    return tb[0];
}

// b0, b1: this lane's coefficients, updated once a sweep from tb; they also
// count the moves (a move changes its coefficient), off the chain.
template <int LD>
__device__ __forceinline__ int phase_sweeps(const float* __restrict__ saa, float2* __restrict__ tb,
                                            int n, float lam, int maxit, float tf, float2 q, float& g0,
                                            float& g1, float& b0, float& b1, unsigned& mv,
                                            bool& conv) {
    const int lane = threadIdx.x & 31;
    const float* __restrict__ col = saa + lane;
    float c0 = col[0], c1 = LD > 32 ? col[32] : 0.f;
    float gk = __shfl_sync(FULL_MASK, g0, 0), dp = 0.f;
    float md;
    unsigned moved = 0;
    // move k; kn is the next one, gs the slot of its gradient
    auto move = [&](int k, int kn, const float& gs) {
        const float gn = __shfl_sync(FULL_MASK, gs, kn);        // (lane kn mod 32)
        float2 qn = tb[kn];
        const float n0 = col[kn * LD], n1 = LD > 32 ? col[kn * LD + 32] : 0.f;
        gk = fmaf(-q.x, dp, gk);
        const float nb = soft_std(gk + q.y, lam);
        dp = nb - q.y;
        tb[k].y = nb;
        if (kn == k) qn.y = nb;
        g0 = fmaf(-c0, dp, g0);
        if (LD > 32) g1 = fmaf(-c1, dp, g1);
        md = max_abs(md, dp);
        c0 = n0;
        c1 = n1;
        q = qn;
        gk = gn;
    };
    int sw = 0;
    while (sw < maxit) {
        ++sw;
        md = 0.f;
        const int n_lo = LD > 32 ? min(n, 32) : n;
#pragma unroll 4
        for (int k = 0; k < n_lo - 1; ++k) move(k, k + 1, g0);
        if (LD > 32) {
#pragma unroll 4
            for (int k = 31; k < n - 1; ++k) move(k, k + 1, g1);
        }
        move(n - 1, 0, g0);
        if (lane < n) {
            const float x = tb[lane].y;
            moved += x != b0;
            b0 = x;
        }
        if (LD > 32 && lane + 32 < n) {
            const float x = tb[lane + 32].y;
            moved += x != b1;
            b1 = x;
        }
        if (md < tf) {
            conv = true;
            break;
        }
    }
    mv = __reduce_add_sync(FULL_MASK, moved);
    return sw;
}

// Active-set phase of the lasso at a fixed lambda: cyclic sweeps (ascending
// coordinate order) over the current support A only, until a sweep moves no
// coefficient by tol or more (at most maxit sweeps).  Lane m holds coordinate
// A_m: its b and g_m = S_jm - sum_{l in A} S_ml b_l; the support's entries of S
// are gathered into shared memory (SupportBlock), and kept from the column's
// last phase when A is the same.  The phase's
// net change of b enters the column's running sums as one change, so the
// chunk skip test stays exact for the coordinates outside A.  Coordinates
// that reach zero leave the support and mark their chunk for a rescan.  One
// move is the phase's critical path: FP32 on the standardised matrix takes
// phase_sweeps; otherwise every lane forms its candidate, one shuffle
// broadcasts the owner's change, and every lane updates its gradient with the
// column of S_AA loaded one move ahead (a zero change adds exact zeros, so no
// lane branches on it).  Returns the sweeps done (0 when A is
// empty or larger than ACT_MAX); `conv` tells whether the last sweep moved
// nothing by tol (true for an empty A, false when A is too large).
template <typename T, bool STD>
__device__ int active_phase(int j, Support<T>& s, const CDArgs<T>& a, T lam, SupportBlock<T>& sb,
                            unsigned long long& moves, ColScan& cs, bool& conv) {
    const int lane = threadIdx.x & 31;
    const int n = s.n;
    conv = n <= ACT_MAX;
    if (n == 0 || n > ACT_MAX) return 0;
    conv = false;
    const int ldp = a.ldp;
    T* __restrict__ saa = sb.saa;
    float2* __restrict__ tb = sb.tb;
    const int my = lane < n ? s.idx[lane] : 0;
    if (!(sb.n == n && __all_sync(FULL_MASK, lane >= n || sb.list[lane] == my))) {
        // lane m reads S_{j A_m}, S_{A_m j} and S_{A_m A_k} for four k at a time
        // (independent loads)
        const T rv = lane < n ? a.SC[(size_t)j * ldp + my] : T(0);
        const T cv = lane < n ? a.SC[(size_t)my * ldp + j] : T(0);
        float tv = 0.f;
        if constexpr (STD) tv = lane < n ? (float)a.diag[my] : 0.f;
#pragma unroll 1
        for (int k0 = 0; k0 < n; k0 += 4) {
            T v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + u;
                v[u] = (k < n && lane < n) ? a.SC[(size_t)my * ldp + s.idx[k]] : T(0);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k0 + u < n) saa[(k0 + u) * ACT_MAX + lane] = v[u];
        }
        sb.row[lane] = rv;
        sb.col[lane] = cv;
        sb.top[lane] = tv;
        sb.list[lane] = my;
        sb.n = n;
    }
    T b = lane < n ? s.val[lane] : T(0);
    const T b_start = b;
    T g = sb.row[lane];
    T skk = T(1);
    if constexpr (!STD) skk = lane < n ? a.diag[my] : T(1);
    __syncwarp();
#pragma unroll 2
    for (int l = 0; l < n; ++l) {
        const T bl = __shfl_sync(FULL_MASK, b, l);
        if (lane < n) g = fma(-saa[l * ACT_MAX + lane], bl, g);
    }
    int sw = 0;
    unsigned mv = 0;
    const float tf = a.tolf;
    if constexpr (STD && sizeof(T) == 4) {
        const float2 first = phase_links<ACT_MAX>(saa, tb, n, b, T(0));
        sw = phase_sweeps<ACT_MAX>(saa, tb, n, lam, a.maxit, tf, first, g, g, b, b, mv, conv);
    } else {
        while (sw < a.maxit) {
            ++sw;
            T md = T(0);
            T c = lane < n ? saa[lane] : T(0);               // column of S_AA for k = 0
            for (int k = 0; k < n; ++k) {
                const int kn = k + 1 < n ? k + 1 : k;
                const T cn = lane < n ? saa[kn * ACT_MAX + lane] : T(0);   // next column
                T nb;
                if constexpr (STD) nb = soft_std(g + b, lam);            // S_kk = 1
                else nb = soft<T>(g + skk * b, lam) / skk;
                const T d = __shfl_sync(FULL_MASK, nb - b, k);
                if (lane == k) b = nb;
                g = fma(-c, d, g);
                md = max_abs(md, d);
                mv += is_move(d);
                c = cn;
            }
            if (below_tol<T>(md, a.tol, tf)) {
                conv = true;
                break;
            }
        }
    }
    moves += mv;
    // the phase enters the running sums as one change: its net l1 size
    const float net = warp_l1_bound(lane < n ? (float)(b - b_start) * sb.top[lane] : 0.f);
    cs.dsum += net * (1.0f + 0x1p-16f);
    ++cs.nmoves;
    // write back, dropping coordinates at zero (the list stays sorted)
    const bool keep = lane < n && b != T(0);
    if (lane < n && b == T(0)) cs.ci[my / CHUNK].maxabs = INFINITY;
    const unsigned km = __ballot_sync(FULL_MASK, keep);
    const int pos = __popc(km & ((1u << lane) - 1u));
    __syncwarp();
    if (keep) {
        s.idx[pos] = my;
        s.val[pos] = b;
    }
    s.n = __popc(km);
    __syncwarp();
    return sw;
}

// sigma_j^2 = S_jj - 2 b'S_.j + b'S b in FP64 over the sorted support (Eq. (14)).
// Every product is formed in FP64 (for FP32 data the product of two FP32
// values is exact in FP64) and every sum is carried in FP64.  FP64 arithmetic
// is scarce on this part and every column runs this step a few times, so the
// FP64 work is kept to a few instructions per lane: the n^2 pairs (u, v) and
// the n terms of b'S_.j are spread over the lanes (pair indices stepped by
// 32 without a divide per pair), each lane adds b_u b_v S_uv and -2 b_u S_uj
// into one FP64 partial, and one FP64 warp sum ends it.
// The entries of S come from the phase's SupportBlock when it was gathered for
// this support (the same values; a sigma step then reads nothing from L2),
// otherwise from S.
template <typename T>
__device__ double residual_quadratic_form_list(int j, const Support<T>& s, const CDArgs<T>& a,
                                               const SupportBlock<T>& sb, double sjj) {
    const int lane = threadIdx.x & 31;
    const int n = s.n;
    const int ldp = a.ldp;
    if (n == 0) return sjj;
    const bool held = sb.n == n && n <= ACT_MAX &&
                      __all_sync(FULL_MASK, lane >= n || sb.list[lane] == s.idx[lane]);
    double acc = 0.0;
    // -2 b_u S_uj for u = lane, lane + 32, ... (-2 b_u is exact in the data precision)
#pragma unroll 1
    for (int u = lane; u < n; u += 32) {
        const T suj = held ? sb.col[u] : a.SC[(size_t)s.idx[u] * ldp + j];
        acc = fma(exact_double(T(-2) * s.val[u]), exact_double(suj), acc);
    }
    const int np = n * n;
    if (lane < np) {
        // pair t = u n + v for t = lane, lane + 32, ...: (u, v) advance by (q, r)
        // (quotients of small integers by a reciprocal: half a unit from an integer
        // is far above its rounding)
        const float rn = __frcp_rn((float)n);
        int u = (int)(((float)lane + 0.5f) * rn), v = lane - u * n;
        const int q = (int)(32.5f * rn), r = 32 - q * n;
#pragma unroll 1
        for (int t = lane; t < np; t += 32) {
            const double bb = exact_double(s.val[u]) * exact_double(s.val[v]);
            const T suv = held ? sb.saa[v * ACT_MAX + u] : a.SC[(size_t)s.idx[u] * ldp + s.idx[v]];
            acc = fma(bb, exact_double(suv), acc);
            u += q;
            v += r;
            if (v >= n) {
                v -= n;
                ++u;
            }
        }
    }
    // the warp sum over the lanes that hold terms (n^2 of them, n >= 1): the
    // others would add exact zeros
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        if (o < np) acc += __shfl_xor_sync(FULL_MASK, acc, o);
    return sjj + __shfl_sync(FULL_MASK, acc, 0);
}

// b_j as the whole dense row j of BT, zeros included (16-byte stores; ldp is a
// multiple of 32): the state of a column that is handed over.
template <typename T>
__device__ __forceinline__ void store_row_lazy(int j, const Support<T>& s, const CDArgs<T>& a) {
    const int lane = threadIdx.x & 31;
    T* brow = a.BT + (size_t)j * a.ldp;
    uint4* q = reinterpret_cast<uint4*>(brow);
    const int nq = a.ldp * (int)sizeof(T) / 16;
#pragma unroll 1
    for (int i = lane; i < nq; i += 32) q[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
#pragma unroll 1
    for (int t = lane; t < s.n; t += 32) brow[s.idx[t]] = s.val[t];
}

// A solved column: b_j as a list in row j of BT and row j of Theta cleared.
template <typename T>
__device__ __forceinline__ void store_solved_lazy(int j, const Support<T>& s, const CDArgs<T>& a) {
    const int lane = threadIdx.x & 31;
    if (a.Theta) clear_theta_row(a.Theta, a.p, j, lane, 32);
    if (s.n > coef_cap(a.ldp)) {
        store_row_lazy<T>(j, s, a);
        if (lane == 0) a.nsup[j] = -1;
        return;
    }
    T* row = a.BT + (size_t)j * a.ldp;
    int* idx = coef_idx(row, a.ldp);
#pragma unroll 1
    for (int t = lane; t < s.n; t += 32) {
        row[t] = s.val[t];
        idx[t] = s.idx[t];
    }
    if (lane == 0) a.nsup[j] = s.n;
}

// The lazy solver's state when it hands column j over: b_j as row j of BT,
// sigma, the last sigma step and the step index, so that the
// block solver continues from this iterate.  Any (b, sigma) is a valid start
// for the coordinate descent, and the hand-over point depends only on the
// column's data, so the result is the same wherever the column is solved.
template <typename T>
__device__ __forceinline__ void hand_over_lazy(int j, const Support<T>& s, const CDArgs<T>& a, double sigma,
                               double s_prev, double f_prev, int r, int status) {
    if (!a.hand) return;
    const int lane = threadIdx.x & 31;
    store_row_lazy<T>(j, s, a);
    if (lane == 0) {
        a.sigma[j] = sigma;
        a.hand[2 * (size_t)j] = s_prev;
        a.hand[2 * (size_t)j + 1] = f_prev;
        a.col_status[j] = COL_HANDED | (status & (COL_NOT_CONVERGED | COL_DEGENERATE)) |
                          (r << COL_STEP_SHIFT);
    }
    __syncwarp();
}

// Algorithm 1 for column j with the lazy gradient.  Returns false when the
// support outgrew the phase or the list (its state is handed over; the caller queues
// the column for the block solver).  HS (single fits) keeps the last sigma step in the
// warp's shared memory instead of registers and takes sigma's sqrt_last here.
template <typename T, bool STD, bool HS = false, int U = 2, int SCAN_G = scan_group<T>()>
__device__ bool solve_column_lazy(int j, unsigned char* wsm, const CDArgs<T>& a, ColCounters& cnt) {
    const int lane = threadIdx.x & 31;
    Support<T> s;
    s.idx = reinterpret_cast<int*>(wsm);
    s.val = reinterpret_cast<T*>(wsm + LAZY_CAP * sizeof(int));
    s.n = 0;
    ColScan cs{reinterpret_cast<ChunkInfo*>(wsm + LAZY_CAP * (sizeof(int) + sizeof(T))), 0.f, 0u};
    double* prev = reinterpret_cast<double*>(cs.ci + num_chunks(a.ldp));   // HS: (sigma, F(sigma)); S_jj; q
    SupportBlock<T> sb;
    sb.saa = reinterpret_cast<T*>(prev + 4);
    sb.row = sb.saa + ACT_MAX * ACT_MAX;
    sb.col = sb.row + ACT_MAX;
    sb.tb = reinterpret_cast<float2*>(sb.col + ACT_MAX);
    sb.list = reinterpret_cast<int*>(sb.tb + (sizeof(T) == 4 ? ACT_MAX : 0));
    sb.top = reinterpret_cast<float*>(sb.list + ACT_MAX);
    sb.n = -1;
    if (lane == 0) prev[2] = exact_double(a.SC[(size_t)j * a.ldp + j]);
    reset_chunks(cs, a.ldp);
    if constexpr (STD) {
        // b = 0: the gradient is row j of S^C, whose chunk maxima the
        // standardisation pass wrote, so the first sweep may skip chunks too
        if (a.chunk_max) {
            const int nch = num_chunks(a.ldp);
            const float* __restrict__ cm = a.chunk_max + (size_t)j * nch;
#pragma unroll 1
            for (int c = lane; c < nch; c += 32) cs.ci[c] = ChunkInfo{cm[c], 0.f, 0u, 0};
        }
    }
    __syncwarp();

    double sigma = 1.0;                                  // sigma^(0) = 1, b = 0
    double s_prev = 0.0, f_prev = 0.0;                   // last (sigma, F(sigma))
    float g_prev = 0.f;                                  // (float)(F(sigma) - sigma) of it
    const unsigned long long sweeps0 = cnt.sweeps;
    int status = COL_OK;
    bool overflow = false;           // the column goes to the block solver
    int r;
    for (r = 0; r < a.maxit; ++r) {
        const T lam = (T)(sigma * a.lambda0);
        bool inner_ok = false;
        for (int m = 0; m < a.maxit; ++m) {
            // converge on the support first; then, if that converged, a
            // sweep over the other coordinates with the support held (its
            // chunks skippable by the bound) decides: the lasso has converged
            // when the support's last sweep and this sweep both moved nothing
            // by tol.  Otherwise a full sweep of every coordinate decides (the
            // stop rule of Algorithm 1).
            bool conv;
            if (s.n > a.ovf_supp) {
                overflow = true;
                break;
            }
            cnt.act_sweeps += active_phase<T, STD>(j, s, a, lam, sb, cnt.act_moves, cs, conv);
            const T md = sweep_column_lazy<T, STD, U, SCAN_G>(j, s, a, lam, cnt.moves, cs, overflow, conv,
                                                   (int)(cnt.sweeps - sweeps0));
            ++cnt.sweeps;
            if (overflow) break;
            if (below_tol<T>(md, a.tol, a.tolf)) {
                inner_ok = true;
                break;
            }
        }
        if (overflow) {
            hand_over_lazy<T>(j, s, a, sigma, HS ? prev[0] : s_prev, HS ? prev[1] : f_prev, r,
                                  status);
            return false;
        }
        if (!inner_ok) status |= COL_NOT_CONVERGED;
        double q = residual_quadratic_form_list<T>(j, s, a, sb, prev[2]);
        // q <= 1e-12 S_jj; a NaN is at the floor too
        const double sjj = prev[2];
        if (may_be_floored(q, sjj)) {
            const double floor2 = 1e-12 * sjj;
            if (!(q > floor2)) {
                q = floor2;
                status |= COL_DEGENERATE;
            }
        }
        const double sn = sqrt_heron(q);
        const double dg = sn - sigma;
        if (lane == 0) prev[3] = q;
        if (below(dg, a.tol)) {
            sigma = sn;
            break;
        }
        double nxt = sn;
        const float g1 = (float)dg;
        if (r > 0 && r + 1 < a.maxit && !(status & COL_DEGENERATE))
            nxt = sigma_step(HS ? prev[0] : s_prev, g_prev, sigma, sn, g1);
        g_prev = g1;
        if constexpr (HS) {
            __syncwarp();
            if (lane == 0) {
                prev[0] = sigma;
                prev[1] = sn;
            }
            __syncwarp();
        } else {
            s_prev = sigma;
            f_prev = sn;
        }
        sigma = nxt;
    }
    if (r == a.maxit) {
        r = a.maxit - 1;
        status |= COL_NOT_CONVERGED;
    }
    store_solved_lazy<T>(j, s, a);
    if (lane == 0) {
        // (the last step's F(sigma) either way)
        if constexpr (HS) sigma = sqrt_last(prev[3], sigma);
        else a.hand[2 * (size_t)j + 1] = prev[3];
        a.sigma[j] = sigma;
        a.col_status[j] = status;
    }
    cnt.outer_max = max(cnt.outer_max, r + 1);
    cnt.max_sw = max(cnt.max_sw, (int)(cnt.sweeps - sweeps0));
    cnt.n_nc += (status & COL_NOT_CONVERGED) != 0;
    cnt.n_deg += (status & COL_DEGENERATE) != 0;
    __syncwarp();
    return true;
}

// ===========================================================================
// Optimality diagnostics of a finished fit (opts.diagnostics).
//
// For column j the returned pair (b_j, sigma_j) solves Algorithm 1's problem
// when the lasso subgradient conditions hold at lambda = lambda0 sigma_j
// (Section 2.1): with g = S_.j - S b_j,
//   g_k = lambda sign(b_k) where b_k != 0,   |g_k| <= lambda where b_k = 0,
// and sigma_j is the fixed point of Eq. (14).  One block per column forms the
// whole gradient in FP64 from the working matrix (row j and the support rows,
// the lazy solver's slices accumulated in FP64) and reports
//  - the largest violation of those conditions relative to lambda;
//  - the relative duality gap (P - D) / P of the lasso subproblem: with
//    rr = S_jj - b'S_.j - b'g (= ||x_j - X b||^2 / n), yr = S_jj - b'S_.j and
//    the dual point s r, s = min(1, lambda / ||g||_inf):
//    P = rr / 2 + lambda ||b||_1, D = s yr - s^2 rr / 2;
//  - a first-order estimate of the error of the column's Theta entries.  The
//    rounding of the working matrix (eps_s per entry, relative) moves each
//    gradient entry by about eps_s (1 + ||b||_2) (independent signs); with
//    the measured gradient residual this is read as a coefficient error
//    (unit diagonal).  sigma moves by the fixed-point residual plus
//    drr / (2 sigma), drr the first-order change of rr: eps_s (1 + ||b||_2)^2
//    from the matrix (at the optimum the change through b is second order)
//    and 2 lambda |A| kkt from a solve that is not exactly optimal.  Then
//    Theta_kj = -b_kj / sigma_j^2, Theta_jj = 1 / sigma_j^2 differentiated.
// ===========================================================================
constexpr int DIAG_CAP = 1024;         // support list of a column
constexpr int DIAG_WARPS = 4;          // warps of a block: the column's chunks in turn.  (One warp
                                       // a column took 92 us for p = 1003, the chain of its
                                       // longest column; four 56.)
static_assert(COEF_CAP <= DIAG_CAP, "a stored list must fit the diagnostics' list");

// Shared memory of a diagnostics block.
struct DiagShared {
    int idx[DIAG_CAP];
    double val[DIAG_CAP];
    double kkt[DIAG_WARPS], gmax[DIAG_WARPS], bg[DIAG_WARPS];
    int ns;
};

// Per-warp maxima of the diagnostics (non-negative doubles), flushed with
// atomicMax on their bits.
struct DiagMax {
    double kkt = 0.0, gap = 0.0, err = 0.0, thmax = 0.0;
};

// (warp 0 of a diagnostics block holds the maxima)
__device__ __forceinline__ void flush_diag(FitCtrl* ctrl, const DiagMax& d) {
    if (threadIdx.x == 0) {
        atomicMax(&ctrl->diag_kkt, dbits(d.kkt));
        atomicMax(&ctrl->diag_gap, dbits(d.gap));
        atomicMax(&ctrl->diag_err, dbits(d.err));
        atomicMax(&ctrl->diag_thmax, dbits(d.thmax));
        atomicAdd(&ctrl->diag_cols, 1u);
    }
}

// By a block of DIAG_WARPS warps; the maxima go to warp 0's `out`.
template <typename T>
__device__ void diagnose_column(int j, DiagShared& sh, const CDArgs<T>& a, double eps_s,
                                DiagMax& out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = a.p, ldp = a.ldp;
    int* __restrict__ idx = sh.idx;
    double* __restrict__ val = sh.val;
    const T* __restrict__ brow = a.BT + (size_t)j * ldp;
    // support of b_j in ascending order: its list, or collected from a dense row
    const int nl = a.nsup ? a.nsup[j] : -1;
    const bool dense = nl < 0;
    if (!dense) {
        const int* __restrict__ src = coef_idx(brow, ldp);
        for (int e = threadIdx.x; e < nl; e += 32 * DIAG_WARPS) {
            idx[e] = src[e];
            val[e] = (double)brow[e];
        }
        if (threadIdx.x == 0) sh.ns = nl;
    } else if (warp == 0) {
        int c = 0;
        for (int c0 = 0; c0 < p; c0 += 32) {
            const int k = c0 + lane;
            const T bk = k < p ? brow[k] : T(0);
            const unsigned bal = __ballot_sync(FULL_MASK, bk != T(0));
            const int pos = c + __popc(bal & ((1u << lane) - 1u));
            if (bk != T(0) && pos < DIAG_CAP) {
                idx[pos] = k;
                val[pos] = (double)bk;
            }
            c += __popc(bal);
        }
        if (lane == 0) sh.ns = c;
    }
    __syncthreads();
    const int ns = sh.ns;
    const bool listed = ns <= DIAG_CAP;
    int e0 = 0;                                       // list: first entry of the chunk
    const double sig = a.sigma[j];
    const double lam = a.lambda0 * sig;
    const T* __restrict__ Sj = a.SC + (size_t)j * ldp;
    double kkt = 0.0, gmax = 0.0, bg = 0.0;
    for (int cb = warp * CHUNK; cb < p; cb += DIAG_WARPS * CHUNK) {
        const int k0 = cb + lane * SCAN_V;
        const bool in = k0 < ldp;
        double acc[SCAN_V] = {0.0, 0.0, 0.0, 0.0};
        if (in) {
            T r[SCAN_V];
            load4g<T>(Sj + k0, r);
#pragma unroll
            for (int t = 0; t < SCAN_V; ++t) acc[t] = (double)r[t];
        }
        if (listed) {
#pragma unroll 4
            for (int e = 0; e < ns; ++e) {
                const double v = val[e];
                if (in) {
                    T r[SCAN_V];
                    load4g<T>(a.SC + (size_t)idx[e] * ldp + k0, r);
#pragma unroll
                    for (int t = 0; t < SCAN_V; ++t) acc[t] = fma(-v, (double)r[t], acc[t]);
                }
            }
        } else {
            for (int l = 0; l < p; ++l) {
                const double v = (double)brow[l];
                if (v != 0.0 && in) {
                    T r[SCAN_V];
                    load4g<T>(a.SC + (size_t)l * ldp + k0, r);
#pragma unroll
                    for (int t = 0; t < SCAN_V; ++t) acc[t] = fma(-v, (double)r[t], acc[t]);
                }
            }
        }
        if (in) {
            double bq[SCAN_V] = {0.0, 0.0, 0.0, 0.0};
            if (dense) {
                T r[SCAN_V];
                load4g<T>(brow + k0, r);
#pragma unroll
                for (int t = 0; t < SCAN_V; ++t) bq[t] = (double)r[t];
            } else {
                while (e0 < ns && idx[e0] < cb) ++e0;
                for (int e = e0; e < ns && idx[e] < cb + CHUNK; ++e) {
                    const int u = idx[e] - k0;
#pragma unroll
                    for (int t = 0; t < SCAN_V; ++t)
                        if (u == t) bq[t] = val[e];
                }
            }
#pragma unroll
            for (int t = 0; t < SCAN_V; ++t) {
                const int k = k0 + t;
                if (k >= p || k == j) continue;
                const double g = acc[t], bk = bq[t];
                const double viol = bk != 0.0 ? fabs(g - copysign(lam, bk)) : fmax(0.0, fabs(g) - lam);
                kkt = fmax(kkt, viol);
                gmax = fmax(gmax, fabs(g));
                if (bk != 0.0) bg = fma(bk, g, bg);
            }
        }
    }
    kkt = warp_max(kkt);
    gmax = warp_max(gmax);
    bg = warp_sum(bg);
    if (lane == 0) {
        sh.kkt[warp] = kkt;
        sh.gmax[warp] = gmax;
        sh.bg[warp] = bg;
    }
    __syncthreads();
    if (warp != 0) return;                            // (the caller's barrier follows)
#pragma unroll
    for (int w = 1; w < DIAG_WARPS; ++w) {
        kkt = fmax(kkt, sh.kkt[w]);
        gmax = fmax(gmax, sh.gmax[w]);
        bg += sh.bg[w];
    }
    double bS = 0.0, l1 = 0.0, l2 = 0.0, bmax = 0.0;
    if (listed) {
        for (int e = lane; e < ns; e += 32) {
            bS = fma(val[e], (double)Sj[idx[e]], bS);
            l1 += fabs(val[e]);
            l2 = fma(val[e], val[e], l2);
            bmax = fmax(bmax, fabs(val[e]));
        }
    } else {
        for (int k = lane; k < p; k += 32) {
            const double v = (double)brow[k];
            bS = fma(v, (double)Sj[k], bS);
            l1 += fabs(v);
            l2 = fma(v, v, l2);
            bmax = fmax(bmax, fabs(v));
        }
    }
    bmax = warp_max(bmax);
    bS = warp_sum(bS);
    l1 = warp_sum(l1);
    l2 = sqrt(warp_sum(l2));
    const double Sjj = (double)Sj[j];
    const double rr = Sjj - bS - bg;
    const double yr = Sjj - bS;
    const double s = gmax > lam ? lam / gmax : 1.0;
    const double P = 0.5 * rr + lam * l1;
    const double D = s * yr - 0.5 * s * s * rr;
    const double gap = P > 0.0 ? fmax(0.0, P - D) / P : 0.0;
    // first-order error of the column's Theta entries
    const double eb = kkt + eps_s * (1.0 + l2);
    const double es = fabs(sig - sqrt(fmax(rr, 0.0))) +
                      (eps_s * (1.0 + l2) * (1.0 + l2) + 2.0 * lam * (double)ns * kkt) / (2.0 * sig);
    const double s2 = sig * sig;
    const double eth = eb / s2 + 2.0 * fmax(1.0, bmax) * es / (s2 * sig);
    out.kkt = fmax(out.kkt, lam > 0.0 ? kkt / lam : kkt);
    out.gap = fmax(out.gap, gap);
    out.err = fmax(out.err, eth);
    out.thmax = fmax(out.thmax, 1.0 / s2);
}

// ===========================================================================
// Block solver for heavy columns.
//
// Algorithm 1 for one column by a whole block of BLK_THREADS threads, for the
// columns whose support is too large for the lazy solver's active-set phase
// (a hub's regression on its neighbours has 40-50 coefficients).  The block
// keeps the whole gradient g_j = S_.j - S b_j and b_j in shared memory:
//  - active-set phase: one warp runs cyclic sweeps over the support A (up to
//    BLK_AMAX coordinates, two per lane, the block S_AA in shared memory)
//    until a sweep moves nothing by tol; then the block forms g afresh from
//    row j and the |A| support rows (no drift accumulates across phases);
//  - working set: after a converged phase one pass over g finds every
//    coordinate outside A that a sweep with A held would move; none ends the
//    lasso at this lambda (that sweep would move nothing), else they join A
//    at b = 0 and the phase runs on the union (while it fits the phase), so
//    coordinates enter the support without an O(p) update per entry;
//  - sweep: the cyclic ascending pass of Algorithm 1 over all coordinates (or
//    with the support held after a converged phase, as in the lazy solver).
//    Every thread tests its coordinates, a block minimum finds the first
//    coordinate whose update changes b, and the rank-1 update
//    g -= S_.k delta (Proposition 2 on S) is applied by the whole block in
//    the same pass that looks for the next mover, so one move costs one pass
//    over g and one barrier;
//  - sigma from Eq. (14) in FP64 over the support (FP64 products), and the
//    safeguarded secant step of the per-column solvers.
// ===========================================================================
constexpr int BLK_THREADS = 512;
constexpr int BLK_WARPS = BLK_THREADS / 32;
constexpr int BLK_AMAX = 64;       // active-set phase: up to 64 coordinates, two per lane
constexpr int BLK_LIST = 1024;     // sorted support list (sigma step, phase, g refresh)
constexpr int BLK_WS_ROUNDS = 16;  // working-set rounds (scan, phase on the union) per inner step
static_assert(LAZY_CAP <= BLK_LIST, "a handed-over support must fit the block solver's list");
static_assert(COEF_CAP <= BLK_LIST, "a stored list must fit the block solver's list");

// Shared memory of the block solver: g and b (ldp each), S_AA, the support
// list, the double-buffered candidate moves of the sweep and the support S_AA
// was gathered for.
template <typename T>
__host__ __device__ constexpr size_t block_smem_bytes(int ldp) {
    return 2 * (size_t)ldp * sizeof(T) + (size_t)BLK_AMAX * BLK_AMAX * sizeof(T) +
           (size_t)BLK_LIST * sizeof(int) + 2 * 2 * (size_t)BLK_THREADS * sizeof(T) +
           (size_t)BLK_AMAX * sizeof(int);
}

// Per-block scratch of the block solver (static shared memory).
struct BlockScratch {
    int red[2][BLK_WARPS];       // block minimum / counts, double-buffered by parity
    double dred[BLK_WARPS];      // FP64 block sums
    int vred[BLK_WARPS];         // scan: coordinates that would move, per warp
    float mred[BLK_WARPS];       // scan: their largest candidate |move|, per warp
    int wcnt[2], wmax[2];        // refresh scan: count and largest |move| (float bits), by parity
    double sig[2];               // the sigma step's F(sigma) and next sigma (warp 0's)
    int sigf;                    // its flags: 1 degenerate, 2 converged
    float bl1;                   // an upper bound of ||b_j||_1 after any phase so far
    int col;
};

// Smallest v over the block (one barrier; `par` alternates the buffer so the
// next call cannot overwrite values still being read).
__device__ __forceinline__ int block_min_int(int v, BlockScratch& sc, int& par) {
    v = __reduce_min_sync(FULL_MASK, v);
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) sc.red[par][warp] = v;
    __syncthreads();
    int m = sc.red[par][0];
#pragma unroll
    for (int w = 1; w < BLK_WARPS; ++w) m = min(m, sc.red[par][w]);
    par ^= 1;
    return m;
}

// Sum of v over the block in a fixed order (deterministic for a fixed block size).
__device__ __forceinline__ double block_sum_d(double v, BlockScratch& sc) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) sc.dred[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < BLK_WARPS; ++w) t += sc.dred[w];
    __syncthreads();
    return t;
}

// Sorted support of b (ascending) into list[0, min(n, BLK_LIST)); returns n.
// Each thread counts the nonzeros of its own contiguous segment of b, a block
// scan gives the segment offsets, and each thread writes its entries.
template <typename T>
__device__ __noinline__ int block_support_list(const T* __restrict__ b, int p, int* __restrict__ list,
                                  BlockScratch& sc, int& par) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int seg = (p + BLK_THREADS - 1) / BLK_THREADS;
    const int k0 = min(p, (int)threadIdx.x * seg), k1 = min(p, k0 + seg);
    int c = 0;
    for (int k = k0; k < k1; ++k) c += b[k] != T(0);
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) sc.red[par][warp] = incl;
    __syncthreads();
    int off = incl - c, total = 0;
#pragma unroll
    for (int w = 0; w < BLK_WARPS; ++w) {
        const int t = sc.red[par][w];
        if (w < warp) off += t;
        total += t;
    }
    par ^= 1;
    for (int k = k0; k < k1 && off < BLK_LIST; ++k)
        if (b[k] != T(0)) list[off++] = k;
    __syncthreads();
    return total;
}

// The nonzero coordinates of src[0, n) (sorted, n <= BLK_AMAX, holding the whole
// support) into list (src itself may be list); returns their number.  A pass over b
// for the support took 12 % of a hub's regression at p = 10000 (5500 cycles each).
template <typename T>
__device__ __forceinline__ int block_filter_list(const T* __restrict__ b, const int* src, int n, int* list,
                                 BlockScratch& sc, int& par) {
    const int lane = threadIdx.x;
    if (lane < 32) {
        const int k0 = lane < n ? src[lane] : 0, k1 = lane + 32 < n ? src[lane + 32] : 0;
        const bool s0 = lane < n && b[k0] != T(0), s1 = lane + 32 < n && b[k1] != T(0);
        const unsigned m0 = __ballot_sync(FULL_MASK, s0), m1 = __ballot_sync(FULL_MASK, s1);
        const unsigned below = (1u << lane) - 1u;
        const int c0 = __popc(m0);
        if (s0) list[__popc(m0 & below)] = k0;
        if (s1) list[c0 + __popc(m1 & below)] = k1;
        if (lane == 0) sc.red[par][0] = c0 + __popc(m1);
    }
    __syncthreads();
    const int m = sc.red[par][0];
    par ^= 1;
    return m;
}

// The scan that certifies a converged support.  A coordinate k != j outside
// the support (b_k = 0) would move in a sweep with the support held exactly
// when its candidate Soft(g_k, lambda) (divided by S_kk without
// standardisation) is nonzero, i.e. |g_k| > lambda; the candidates are formed
// as the sweep forms them.  Writes the sorted union of the support and those
// coordinates into list[0, min(n, BLK_LIST)) and returns n; nv is the number
// of coordinates that would move and mv the largest |candidate| among them
// (each taken as if it moved first).  Same segment layout as
// block_support_list; the block's counts are read before its last barrier,
// so the single-buffered vred / mred can be written by the next call.
template <typename T, bool STD>
__device__ __forceinline__ bool scan_member(int k, int j, const T* __restrict__ g,
                                            const T* __restrict__ b, const CDArgs<T>& a, T lam,
                                            T& nb) {
    const T bk = b[k];
    nb = T(0);
    if (bk != T(0)) return true;
    if (k == j) return false;
    if constexpr (STD) nb = soft<T>(g[k] + bk, lam);                         // S_kk = 1
    else nb = soft<T>(g[k] + a.diag[k] * bk, lam) / a.diag[k];
    return nb != T(0);
}

template <typename T, bool STD>
__device__ __noinline__ int block_scan_list(int j, const T* __restrict__ g, const T* __restrict__ b,
                               const CDArgs<T>& a, T lam, int* __restrict__ list, BlockScratch& sc,
                               int& par, int& nv, float& mv) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int p = a.p;
    const int seg = (p + BLK_THREADS - 1) / BLK_THREADS;
    const int k0 = min(p, (int)threadIdx.x * seg), k1 = min(p, k0 + seg);
    int c = 0, v = 0;
    float m = 0.f;
    for (int k = k0; k < k1; ++k) {
        T nb;
        if (scan_member<T, STD>(k, j, g, b, a, lam, nb)) {
            ++c;
            if (nb != T(0)) {
                ++v;
                m = fmaxf(m, fabsf((float)nb));
            }
        }
    }
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(FULL_MASK, incl, o);
        if (lane >= o) incl += u;
    }
    const int vw = __reduce_add_sync(FULL_MASK, v);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(FULL_MASK, m, o));
    if (lane == 31) sc.red[par][warp] = incl;
    if (lane == 0) {
        sc.vred[warp] = vw;
        sc.mred[warp] = m;
    }
    __syncthreads();
    int off = incl - c, total = 0, vt = 0;
    float mt = 0.f;
#pragma unroll
    for (int w = 0; w < BLK_WARPS; ++w) {
        const int t = sc.red[par][w];
        if (w < warp) off += t;
        total += t;
        vt += sc.vred[w];
        mt = fmaxf(mt, sc.mred[w]);
    }
    par ^= 1;
    for (int k = k0; k < k1 && off < BLK_LIST; ++k) {
        T nb;
        if (scan_member<T, STD>(k, j, g, b, a, lam, nb)) list[off++] = k;
    }
    __syncthreads();
    nv = vt;
    mv = mt;
    return total;
}

// Whether k is one of the sorted list[0, n) (binary search).
__device__ __forceinline__ bool list_contains(const int* __restrict__ list, int n, int k) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (list[mid] < k) lo = mid + 1;
        else hi = mid;
    }
    return lo < n && list[lo] == k;
}

// The scan of a converged support, folded into the gradient refresh: while
// g is formed, every coordinate k != j outside list[0, n) with b_k = 0 whose
// candidate Soft(g_k, lambda) (divided by S_kk without standardisation) is
// nonzero, i.e. which a sweep with the support held would move, is counted
// into sc.wcnt[wp] and, while there is room, appended to vlist (in no
// particular order); sc.wmax[wp] keeps the largest |candidate| (as the bits
// of a non-negative float).  Thread 0 clears the other parity's pair for
// the next scan: that pair was last read before a barrier that every thread
// has passed since.
struct RefreshScan {
    int* vlist;
    int vcap;
    int wp;
};

// Bounds of the gradient by chunk (standardised matrix), kept from one
// refresh with a scan to the next: ub[c] >= |g_k| for every k != j of chunk c
// that was neither j nor in the support at the last one, `prev[0, nprev)` holds that support's
// list, and a phase leaves the change of each of its coordinates in dl.  With
// |S^C_lk| <= cmax[l][c], chunk c grows by at most sum_l dl_l cmax[l][c]; while
// that stays below lambda (with the margins of chunk_skippable) no coordinate at
// zero in it would move, so the refresh leaves the chunk out: the scan finds the same
// coordinates.  A coordinate that has reached zero since opens its chunk.  What reads all of g
// (block_sweep, block_scan_list) has it formed whole first.  Of 79 chunks the
// refreshes of a hub's regression (p = 10000, 49 coefficients) form 78, 78, 11, 79, 2,
// 1, 2 and 0; a whole one takes 50 kcycles, rows from L2 and DRAM.  With the
// support's list kept, S_AA gathered by the block and the sigma step's FP64 in one
// warp, that fit takes 926 us instead of 989, and 256 mixed fits 1897 instead of 1935.
struct ChunkBounds {
    float* ub;
    int* prev;
    float* dl;
    int nprev;
    bool valid;
};
constexpr int BLK_MAX_CHUNKS = 1024;       // chunks the bounds have room for

// g = S_.j - sum_{l in A} S_.l b_l (block-wide), A = list[0, n): over the whole row,
// or over the chunks that `cb` cannot leave out.  Warp w takes chunks w, w + 16, ...,
// QG at once, and reads R support rows for each, so
// QG * R independent loads are in flight; the products are accumulated in
// the order of the list.  With `scan` the refresh also scans (RefreshScan), and
// with cb it leaves the bounds of the chunks that it forms; plist[0, np) are the
// coordinates of the phase before it.
template <typename T, bool STD>
__device__ __noinline__ void block_form_gradient(int j, T* __restrict__ g, const T* __restrict__ b,
                                    const int* __restrict__ list, int n, const CDArgs<T>& a,
                                    bool scan, T lam, BlockScratch& sc, RefreshScan ws,
                                    const ChunkBounds* cb, const int* __restrict__ plist, int np) {
    static_assert(CHUNK == 128, "a warp's quads are one chunk");
    constexpr int QG = sizeof(T) == 4 ? 2 : 1, R = 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ldp = a.ldp, nch = num_chunks(ldp);
    const T* __restrict__ Sj = a.SC + (size_t)j * ldp;
    if (scan) {
        if (threadIdx.x == 0) {
            sc.wcnt[ws.wp ^ 1] = 0;
            sc.wmax[ws.wp ^ 1] = 0;
        }
    }
    for (int base = warp; base < nch; base += 32 * BLK_WARPS) {
        // the warp's chunks base + 16 i to be formed, i < 32
        const int cnt = min(32, (nch - base + BLK_WARPS - 1) / BLK_WARPS);
        unsigned open = cnt == 32 ? FULL_MASK : (1u << cnt) - 1u;
        if (STD && cb && cb->valid) {
            const float d0 = lane < np ? cb->dl[lane] : 0.f, d1 = lane + 32 < np ? cb->dl[lane + 32] : 0.f;
            const float* r0 = a.chunk_max + (size_t)(lane < np ? plist[lane] : j) * nch + base;
            const float* r1 = a.chunk_max + (size_t)(lane + 32 < np ? plist[lane + 32] : j) * nch + base;
            const float top = (float)lam - (2.0f + 2.0f * sc.bl1) * 0x1p-14f;
            unsigned keep = 0u;
            for (int i0 = 0; i0 < cnt; i0 += 4) {
                float x[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    x[i] = i0 + i < cnt ? d0 * r0[(i0 + i) * BLK_WARPS] + d1 * r1[(i0 + i) * BLK_WARPS]
                                        : 0.f;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if (i0 + i >= cnt) break;
                    const int c = base + (i0 + i) * BLK_WARPS;
                    const float u = (cb->ub[c] + warp_l1_bound(x[i]) * (1.0f + 0x1p-10f)) * (1.0f + 0x1p-20f);
                    __syncwarp();
                    if (u < top) {
                        if (lane == 0) cb->ub[c] = u;
                        keep |= 1u << (i0 + i);
                    }
                }
            }
            // chunks of coordinates that have reached zero
            unsigned left = 0u;
            for (int e = lane; e < cb->nprev; e += 32) {
                const int k = cb->prev[e], i = k / CHUNK - base;
                if (b[k] == T(0) && i >= 0 && i % BLK_WARPS == 0 && i / BLK_WARPS < cnt)
                    left |= 1u << (i / BLK_WARPS);
            }
            keep &= ~__reduce_or_sync(FULL_MASK, left);
            open &= ~keep;
        }
        while (open) {
            int k0[QG];
#pragma unroll
            for (int u = 0; u < QG; ++u) {
                k0[u] = ldp;                                   // no chunk: nothing is read
                if (open) {
                    k0[u] = (base + (__ffs(open) - 1) * BLK_WARPS) * CHUNK + 4 * lane;
                    open &= open - 1u;
                }
            }
            T acc[QG][4];
#pragma unroll
            for (int u = 0; u < QG; ++u)
                if (k0[u] < ldp) load4g<T>(Sj + k0[u], acc[u]);
            int e = 0;
            for (; e + R <= n; e += R) {
                T r[R][QG][4];
#pragma unroll
                for (int v = 0; v < R; ++v) {
                    const T* __restrict__ row = a.SC + (size_t)list[e + v] * ldp;
#pragma unroll
                    for (int u = 0; u < QG; ++u)
                        if (k0[u] < ldp) load4g<T>(row + k0[u], r[v][u]);
                }
#pragma unroll
                for (int v = 0; v < R; ++v) {
                    const T bv = b[list[e + v]];
#pragma unroll
                    for (int u = 0; u < QG; ++u)
#pragma unroll
                        for (int t = 0; t < 4; ++t) acc[u][t] = fma(-bv, r[v][u][t], acc[u][t]);
                }
            }
            for (; e < n; ++e) {
                const T* __restrict__ row = a.SC + (size_t)list[e] * ldp;
                const T bv = b[list[e]];
#pragma unroll
                for (int u = 0; u < QG; ++u) {
                    if (k0[u] < ldp) {
                        T r[4];
                        load4g<T>(row + k0[u], r);
#pragma unroll
                        for (int t = 0; t < 4; ++t) acc[u][t] = fma(-bv, r[t], acc[u][t]);
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < QG; ++u) {
                if (k0[u] < ldp)
#pragma unroll
                    for (int t = 0; t < 4; ++t) g[k0[u] + t] = acc[u][t];
            }
            if (scan) {
#pragma unroll
                for (int u = 0; u < QG; ++u) {
                    float top = 0.f;
                    if (k0[u] < a.p) {
                        T bq[4];
                        load4<T>(b + k0[u], bq);
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const int k = k0[u] + t;
                            if (k < a.p && k != j && bq[t] == T(0)) {
                                T nb;
                                if constexpr (STD) nb = soft<T>(acc[u][t] + bq[t], lam);     // S_kk = 1
                                else nb = soft<T>(acc[u][t] + a.diag[k] * bq[t], lam) / a.diag[k];
                                if (STD) top = fmaxf(top, fabsf((float)acc[u][t]));
                                if (nb != T(0) && !list_contains(list, n, k)) {
                                    const int slot = atomicAdd(&sc.wcnt[ws.wp], 1);
                                    if (slot < ws.vcap) ws.vlist[slot] = k;
                                    atomicMax(&sc.wmax[ws.wp], __float_as_int(fabsf((float)nb)));
                                }
                            }
                        }
                    }
                    if (STD && cb) {
                        // lane 0 holds the chunk's first coordinate, below ldp when there is a chunk
                        const unsigned m = __reduce_max_sync(FULL_MASK, __float_as_uint(top));
                        if (lane == 0 && k0[u] < ldp) cb->ub[k0[u] / CHUNK] = __uint_as_float(m);
                    }
                }
            }
        }
    }
}

// The sorted union of list[0, n) (sorted) and vlist[0, nv) (distinct, not in
// the list, in any order) into u[0, n + nv), by warp 0 (n + nv <= BLK_AMAX):
// an entry's place is the number of entries of both lists below it.
__device__ inline void warp_union(const int* __restrict__ list, int n, const int* __restrict__ vlist,
                           int nv, int* __restrict__ u) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int e = lane + 32 * h;
        int x = INT_MAX, cv = 0;
        if (e < n) x = list[e];
        int y = INT_MAX, ry = 0;
        if (e < nv) y = vlist[e];
        for (int t = 0; t < nv; ++t) {
            const int w = vlist[t];
            cv += w < x;
            ry += w < y;
        }
        if (e < n) u[e + cv] = x;
        if (e < nv) {
            int lo = 0, hi = n;                       // entries of the list below y
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (list[mid] < y) lo = mid + 1;
                else hi = mid;
            }
            u[ry + lo] = y;
        }
    }
    __syncwarp();
}

// S_AA of A = list[0, n), n <= BLK_AMAX, by the whole block: warp w gathers rows
// w, w + 16, ... with all of its loads in flight (one warp alone took 67 of a
// hub's 800 kcycles at p = 10000); zero outside the n x n block so the idle slots
// stay finite.  Kept from the last phase when the support is the same
// (saa_list, saa_n; the same in every thread).
template <typename T>
__device__ __forceinline__ void block_gather_saa(const int* __restrict__ list, int n, const CDArgs<T>& a,
                                                 T* __restrict__ saa, int* __restrict__ saa_list,
                                                 int& saa_n) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (__syncthreads_and(saa_n == n && (tid >= n || saa_list[tid] == list[tid]))) return;
    constexpr int NR = BLK_AMAX / BLK_WARPS;
    const int m0 = lane, m1 = lane + 32;
    const int l0 = m0 < n ? list[m0] : 0, l1 = m1 < n ? list[m1] : 0;
    T v0[NR], v1[NR];
#pragma unroll
    for (int u = 0; u < NR; ++u) {
        const int k = warp + u * BLK_WARPS;
        const T* __restrict__ row = a.SC + (size_t)(k < n ? list[k] : 0) * a.ldp;
        v0[u] = (k < n && m0 < n) ? row[l0] : T(0);
        v1[u] = (k < n && m1 < n) ? row[l1] : T(0);
    }
#pragma unroll
    for (int u = 0; u < NR; ++u) {
        const int k = warp + u * BLK_WARPS;
        saa[k * BLK_AMAX + m0] = v0[u];
        saa[k * BLK_AMAX + m1] = v1[u];
    }
    if (tid < n) saa_list[tid] = list[tid];
    saa_n = n;
    __syncthreads();
}

// Active-set phase of the block solver, run by warp 0 on A = list[0, n),
// n <= BLK_AMAX: lane m holds coordinates A_m and A_{m+32}.  Reads and writes
// b for the coordinates of A; g is formed afresh by the caller afterwards.
// Returns the sweeps done; conv tells whether the last one moved nothing by tol.
// One move is the critical path of the phase (phase_sweeps for FP32 on the
// standardised matrix; otherwise the owner's change is broadcast by one
// shuffle, and every lane updates its two gradients with the column of S_AA
// loaded one move ahead).  A zero change adds exact zeros, so no lane branches
// on it.
template <typename T, bool STD>
__device__ int block_active_phase(int j, T* __restrict__ b, const int* __restrict__ list, int n,
                                  const CDArgs<T>& a, T lam, const T* __restrict__ saa,
                                  float2* __restrict__ tb, float* __restrict__ dl, BlockScratch& sc,
                                  unsigned long long& moves, bool& conv) {
    const int lane = threadIdx.x & 31;
    const int ldp = a.ldp;
    const int m0 = lane, m1 = lane + 32;
    const bool h0 = m0 < n, h1 = m1 < n;
    T b0 = h0 ? b[list[m0]] : T(0), b1 = h1 ? b[list[m1]] : T(0);
    T g0 = h0 ? a.SC[(size_t)j * ldp + list[m0]] : T(0);
    T g1 = h1 ? a.SC[(size_t)j * ldp + list[m1]] : T(0);
    const T b0_start = b0, b1_start = b1;
    T s0 = T(1), s1 = T(1);
    if constexpr (!STD) {
        if (h0) s0 = a.diag[list[m0]];
        if (h1) s1 = a.diag[list[m1]];
    }
    __syncwarp();
    for (int l = 0; l < n; ++l) {
        const T bl = __shfl_sync(FULL_MASK, l < 32 ? b0 : b1, l & 31);
        g0 = fma(-saa[l * BLK_AMAX + m0], bl, g0);
        g1 = fma(-saa[l * BLK_AMAX + m1], bl, g1);
    }
    conv = false;
    int sw = 0;
    unsigned mv = 0;
    const float tf = a.tolf;
    if constexpr (STD && sizeof(T) == 4) {
        const float2 first = phase_links<BLK_AMAX>(saa, tb, n, b0, b1);
        sw = phase_sweeps<BLK_AMAX>(saa, tb, n, lam, a.maxit, tf, first, g0, g1, b0, b1, mv, conv);
    } else {
        while (sw < a.maxit) {
            ++sw;
            T md = T(0);
            T c0 = saa[m0], c1 = saa[m1];                 // column of S_AA for k = 0
            for (int k = 0; k < n; ++k) {
                const int kn = k + 1 < n ? k + 1 : k;
                const T n0 = saa[kn * BLK_AMAX + m0], n1 = saa[kn * BLK_AMAX + m1];   // next column
                const bool hi = k >= 32;
                const T gk = hi ? g1 : g0, bk = hi ? b1 : b0;
                T nb;
                if constexpr (STD) {
                    nb = soft_std(gk + bk, lam);                     // S_kk = 1
                } else {
                    const T sk = hi ? s1 : s0;
                    nb = soft<T>(gk + sk * bk, lam) / sk;
                }
                const T d = __shfl_sync(FULL_MASK, nb - bk, k & 31);
                if (lane == (k & 31)) {
                    if (hi) b1 = nb;
                    else b0 = nb;
                }
                g0 = fma(-c0, d, g0);
                g1 = fma(-c1, d, g1);
                md = max_abs(md, d);
                mv += is_move(d);
                c0 = n0;
                c1 = n1;
            }
            if (below_tol<T>(md, a.tol, tf)) {
                conv = true;
                break;
            }
        }
    }
    moves += mv;
    if (h0) b[list[m0]] = b0;
    if (h1) b[list[m1]] = b1;
    dl[m0] = fabsf((float)(b0 - b0_start));                 // ChunkBounds
    dl[m1] = fabsf((float)(b1 - b1_start));
    const float l1 = warp_l1_bound((float)b0) + warp_l1_bound((float)b1);
    if (lane == 0) sc.bl1 = fmaxf(sc.bl1, l1);
    return sw;
}

// One sweep of the block solver (cyclic ascending, k != j; with `frozen` the
// coordinates of the support keep their values).  Returns max |delta b|.
// cand holds the candidate moves (new b, delta) of every thread, two buffers.
// Out of line on the standardised matrix (inlined it took a hub's regression at p = 10000
// from 932 to 979 us), with what it reads of its arguments in registers: through the
// references each move of a sweep was 10 % slower (p = 700, more than 64 coefficients a column,
// 17.3 against 15.3 ms a fit).  Without standardisation inline (45.5 against 45.0).
template <typename T, bool STD>
__device__ __forceinline__ T block_sweep_body(int j, T* __restrict__ g, T* __restrict__ b, const CDArgs<T>& a, T lam,
                         bool frozen, T* __restrict__ cand, unsigned long long& moves,
                         BlockScratch& sc, int& par0, int sweep_idx) {
    const int tid = threadIdx.x;
    const int p = a.p, ldp = a.ldp;
    const T* __restrict__ SC = a.SC;
    const T* __restrict__ diag = a.diag;
    const bool note = a.rows_moved != nullptr;
    int par = par0;
    unsigned n_moves = 0;
    T maxd = T(0);
    int ks = -1;                      // the move of the last pass, applied in this pass
    T delta = T(0);
    for (;;) {
        const T* __restrict__ srow = SC + (size_t)(ks < 0 ? 0 : ks) * ldp;
        T* __restrict__ cb = cand + (size_t)par * 2 * BLK_THREADS;
        int kmin = INT_MAX;
        // the thread's quads q0, q0 + BLK_THREADS, ... in groups of G, the
        // group's S-row loads issued together
        constexpr int G = sizeof(T) == 4 ? 4 : 2;
        for (int q0 = tid; 4 * q0 < ldp; q0 += G * BLK_THREADS) {
            T r[G][4];
            if (ks >= 0) {
#pragma unroll
                for (int u = 0; u < G; ++u) {
                    const int k0 = 4 * (q0 + u * BLK_THREADS);
                    if (k0 < ldp) load4g<T>(srow + k0, r[u]);
                }
            }
#pragma unroll
          for (int u = 0; u < G; ++u) {
            const int k0 = 4 * (q0 + u * BLK_THREADS);
            if (k0 >= ldp) break;
            T gv[4];
            load4<T>(g + k0, gv);
            if (ks >= 0) {            // rank-1 update g -= S_.ks delta (Proposition 2)
#pragma unroll
                for (int t = 0; t < 4; ++t) gv[t] = fma(-delta, r[u][t], gv[t]);
#pragma unroll
                for (int t = 0; t < 4; ++t) g[k0 + t] = gv[t];
            }
            if (kmin == INT_MAX && k0 + 3 > ks && k0 < p) {
                T bv[4];
                load4<T>(b + k0, bv);
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    const int k = k0 + t;
                    if (kmin == INT_MAX && k > ks && k < p && k != j && !(frozen && bv[t] != T(0))) {
                        T nb;
                        if constexpr (STD) {
                            nb = soft<T>(gv[t] + bv[t], lam);                 // S_kk = 1
                        } else {
                            const T skk = diag[k];
                            nb = soft<T>(gv[t] + skk * bv[t], lam) / skk;     // Soft(c, lambda)/S_kk
                        }
                        if (nb != bv[t]) {
                            kmin = k;
                            cb[tid] = nb;
                            cb[BLK_THREADS + tid] = nb - bv[t];
                        }
                    }
                }
            }
          }
        }
        const int kb = block_min_int(kmin, sc, par);    // barrier: g updated, candidates visible
        if (kb == INT_MAX) break;
        const int owner = (kb >> 2) % BLK_THREADS;      // the thread whose quads hold kb
        delta = cb[BLK_THREADS + owner];
        if (tid == owner) {
            b[kb] = cb[owner];
            if (note) note_row_moved(a, sweep_idx, kb);
        }
        maxd = fmax(maxd, fabs(delta));
        ++n_moves;
        ks = kb;
    }
    moves += n_moves;
    par0 = par;
    return maxd;
}

template <typename T>
__device__ __noinline__ T block_sweep_std(int j, T* __restrict__ g, T* __restrict__ b, const CDArgs<T>& a,
                                          T lam, bool frozen, T* __restrict__ cand,
                                          unsigned long long& moves, BlockScratch& sc, int& par,
                                          int sweep_idx) {
    return block_sweep_body<T, true>(j, g, b, a, lam, frozen, cand, moves, sc, par, sweep_idx);
}
template <typename T, bool STD>
__device__ __forceinline__ T block_sweep(int j, T* __restrict__ g, T* __restrict__ b, const CDArgs<T>& a,
                                         T lam, bool frozen, T* __restrict__ cand,
                                         unsigned long long& moves, BlockScratch& sc, int& par,
                                         int sweep_idx) {
    if constexpr (STD) return block_sweep_std<T>(j, g, b, a, lam, frozen, cand, moves, sc, par, sweep_idx);
    else return block_sweep_body<T, false>(j, g, b, a, lam, frozen, cand, moves, sc, par, sweep_idx);
}

// sigma_j^2 = S_jj - 2 b'S_.j + b'S b in FP64 over the support list (block-wide),
// FP64 products; a support longer than the list takes the rows from b itself.
template <typename T>
__device__ __noinline__ double block_quadratic_form(int j, const T* __restrict__ b, const int* __restrict__ list,
                                       int n, const CDArgs<T>& a, BlockScratch& sc) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ldp = a.ldp, p = a.p;
    double lin = 0.0, quad = 0.0;
    if (n <= BLK_LIST) {
        for (int u = warp; u < n; u += BLK_WARPS) {
            const int ku = list[u];
            const T* __restrict__ row = a.SC + (size_t)ku * ldp;
            double part = 0.0;
            for (int v = lane; v < n; v += 32) {
                const int kv = list[v];
                part = fma((double)b[kv], (double)row[kv], part);
            }
            quad = fma((double)b[ku], part, quad);
            if (lane == 0) lin = fma((double)b[ku], (double)row[j], lin);
        }
    } else {
        for (int u = warp; u < p; u += BLK_WARPS) {
            const T bu = b[u];
            if (bu == T(0)) continue;
            const T* __restrict__ row = a.SC + (size_t)u * ldp;
            double part = 0.0;
            for (int v = lane; v < p; v += 32)
                if (b[v] != T(0)) part = fma((double)b[v], (double)row[v], part);
            quad = fma((double)bu, part, quad);
            if (lane == 0) lin = fma((double)bu, (double)row[j], lin);
        }
    }
    lin = block_sum_d(lin, sc);
    quad = block_sum_d(quad, sc);
    return (double)a.SC[(size_t)j * ldp + j] - 2.0 * lin + quad;
}

// sigma_j^2 = S_jj - 2 b'S_.j + b'S b (Eq. (14)) in FP64 from the block
// S_AA in shared memory, when the support lies in the list A it was
// gathered for (A = saa_list[0, na), sorted; saa[k BLK_AMAX + m] = S_{A_k A_m}):
// b is zero on A outside the support, and the zero terms add nothing.
// Returns false (nothing computed) when some support coordinate is not in A;
// q is valid in warp 0.  The FP64 pipe (16 cycles a warp's instruction) bounds this, so
// the products are formed by BLK_QWARPS warps, warp w taking the rows k = w,
// w + 4, ... of S_AA and each lane two of its entries, only these warps' sums are
// formed, and one warp adds them up: with all 16 warps in each of these steps
// a sigma step took 12 of a hub's 850 kcycles (p = 10000, six steps).
constexpr int BLK_QWARPS = 4;
template <typename T>
__device__ __noinline__ bool block_quadratic_form_saa(int j, const T* __restrict__ b, int nsupp,
                                         const int* __restrict__ saa_list, int na,
                                         const T* __restrict__ saa, const CDArgs<T>& a,
                                         BlockScratch& sc, double& q) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int tid = threadIdx.x;
    if (na <= 0 || na > BLK_AMAX || nsupp > na) return false;
    const int v0 = lane, v1 = lane + 32;
    // S_kj and S_jj (warp 0), on their way during the products
    T s0 = T(0), s1 = T(0), sjj = T(0);
    if (warp == 0) {
        if (v0 < na) s0 = a.SC[(size_t)saa_list[v0] * a.ldp + j];
        if (v1 < na) s1 = a.SC[(size_t)saa_list[v1] * a.ldp + j];
        sjj = a.SC[(size_t)j * a.ldp + j];
    }
    const int inA = __syncthreads_count(tid < na && b[saa_list[tid]] != T(0));
    if (inA != nsupp) return false;
    if (warp < BLK_QWARPS) {
        const T b0 = v0 < na ? b[saa_list[v0]] : T(0), b1 = v1 < na ? b[saa_list[v1]] : T(0);
        const double bv0 = exact_double(b0), bv1 = exact_double(b1);
        double acc = 0.0;
        if (na <= 32) {
#pragma unroll 4
            for (int k = warp; k < na; k += BLK_QWARPS)     // b_k sum_m S_km b_m
                acc = fma(exact_double(b[saa_list[k]]), bv0 * exact_double(saa[k * BLK_AMAX + v0]), acc);
        } else {
#pragma unroll 4
            for (int k = warp; k < na; k += BLK_QWARPS)
                acc = fma(exact_double(b[saa_list[k]]),
                          fma(bv1, exact_double(saa[k * BLK_AMAX + v1]),
                              bv0 * exact_double(saa[k * BLK_AMAX + v0])), acc);
        }
        if (warp == 0) {                                    // -2 b_k S_kj
            acc = fma(exact_double(T(-2) * b0), exact_double(s0), acc);
            if (na > 32) acc = fma(exact_double(T(-2) * b1), exact_double(s1), acc);
        }
        acc = warp_sum(acc);
        if (lane == 0) sc.dred[warp] = acc;
    }
    __syncthreads();
    if (warp == 0) {
        double t = exact_double(sjj);
#pragma unroll
        for (int w = 0; w < BLK_QWARPS; ++w) t += sc.dred[w];
        q = t;
    }
    return true;
}

// Algorithm 1 for column j by the whole block (see above).  Writes b_j (row j of
// BT), sigma_j and the column status.  Counters are kept
// identically by every thread; the caller flushes thread 0's.
template <typename T, bool STD>
__device__ void solve_column_block(int j, unsigned char* smem, const CDArgs<T>& a,
                                   ColCounters& cnt, BlockScratch& sc) {
    const int tid = threadIdx.x;
    const int ldp = a.ldp;
    T* g = reinterpret_cast<T*>(smem);
    T* b = g + ldp;
    T* saa = b + ldp;
    int* list = reinterpret_cast<int*>(saa + BLK_AMAX * BLK_AMAX);
    T* cand = reinterpret_cast<T*>(list + BLK_LIST);
    int* saa_list = reinterpret_cast<int*>(cand + 2 * 2 * BLK_THREADS);   // support of S_AA
    // the candidate buffers are idle between sweeps: the working set's union
    // and the refresh scan's coordinates live there
    int* ubuf = reinterpret_cast<int*>(cand);
    int* vlist = ubuf + BLK_AMAX;
    // the phase's links and coefficients too (2 KB of the buffers' 8 KB at most)
    float2* tb = reinterpret_cast<float2*>(vlist + BLK_AMAX);
    // and, between sweeps, the bounds of the gradient's chunks (5 KB)
    ChunkBounds cb;
    cb.prev = reinterpret_cast<int*>(tb) + 2048 / sizeof(int);
    cb.dl = reinterpret_cast<float*>(cb.prev + BLK_AMAX);
    cb.ub = cb.dl + BLK_AMAX;
    static_assert(4 * BLK_AMAX * sizeof(int) + 2048 + BLK_MAX_CHUNKS * sizeof(float) <=
                  2 * 2 * BLK_THREADS * sizeof(float), "the bounds share the candidate buffers");
    cb.nprev = 0;
    cb.valid = false;
    const int nch = num_chunks(ldp);
    const bool bounds = STD && a.chunk_max && nch <= BLK_MAX_CHUNKS;
    bool gfull = true;                                    // every chunk of g is up to date
    int saa_n = -1;                                       // no S_AA gathered yet
    int par = 0;
    int wp = 0;                                           // parity of the refresh scan's counters
    // a column the lazy solver handed over continues from its iterate
    const int st0 = a.hand ? a.col_status[j] : COL_OK;
    const bool warm = (st0 & COL_HANDED) != 0;
    {
        const T* __restrict__ Sj = a.SC + (size_t)j * ldp;
        const T* __restrict__ brow = a.BT + (size_t)j * ldp;
        for (int k = tid; k < ldp; k += BLK_THREADS) {
            g[k] = Sj[k];                                 // g = S_.j  (b = 0)
            b[k] = warm ? brow[k] : T(0);
        }
        if (tid == 0) {
            sc.wcnt[0] = sc.wcnt[1] = 0;
            sc.wmax[0] = sc.wmax[1] = 0;
            sc.bl1 = 0.f;
        }
        if (bounds && !warm) {                            // b = 0: the row's chunk maxima
            for (int c = tid; c < nch; c += BLK_THREADS) cb.ub[c] = a.chunk_max[(size_t)j * nch + c];
            cb.valid = true;
        }
    }
    __syncthreads();
    double sigma = 1.0;                                   // sigma^(0) = 1
    double s_prev = 0.0, f_prev = 0.0;                    // last (sigma, F(sigma))
    int status = COL_OK;
    int r0 = 0;
    bool stale = false;                                   // g is not yet S_.j - S b
    // list[0, nl) (or its first BLK_LIST) holds the support, and nothing else if `exact`;
    // nl = -1 when that is not known
    int nl = warm ? -1 : 0;
    bool exact = true;
    auto support = [&]() {
        if (nl < 0) nl = block_support_list<T>(b, a.p, list, sc, par);
        else if (!exact) nl = block_filter_list<T>(b, list, nl, list, sc, par);
        exact = true;
        return nl;
    };
    // the chunks that refreshes have left out (the support is then one of a phase)
    auto form_all = [&]() {
        block_form_gradient<T, STD>(j, g, b, list, nl, a, false, T(0), sc, RefreshScan{vlist, 0, wp},
                                    nullptr, list, 0);
        __syncthreads();
        gfull = true;
    };
    if (warm) {
        sigma = a.sigma[j];
        s_prev = a.hand[2 * (size_t)j];
        f_prev = a.hand[2 * (size_t)j + 1];
        status = st0 & (COL_NOT_CONVERGED | COL_DEGENERATE);
        r0 = st0 >> COL_STEP_SHIFT;
        stale = true;
    }
    const unsigned long long sweeps0 = cnt.sweeps;
    const double floor2 = 1e-12 * (double)a.SC[(size_t)j * ldp + j];
    int r;
    for (r = r0; r < a.maxit; ++r) {
        const T lam = (T)(sigma * a.lambda0);
        bool inner_ok = false;
        int rounds = 0;              // working-set rounds at this lambda
        bool uni = false;            // ubuf[0, nu) holds the union for the next phase
        int nu = 0;
        for (int m = 0; m < a.maxit; ++m) {
            // converge on the support first (when it fits the phase), then a
            // sweep with the support held decides; otherwise a full sweep
            // decides (Algorithm 1's stop), as in the lazy solver
            int n = uni ? nu : support();
            const int* plist = uni ? ubuf : list;
            const int np = n;
            bool conv = n == 0;
            const bool phase = n > 0 && n <= BLK_AMAX;
            if (phase) {
                int sw = 0;
                bool c = false;
                block_gather_saa<T>(plist, n, a, saa, saa_list, saa_n);
                if (tid < 32) sw = block_active_phase<T, STD>(j, b, plist, n, a, lam, saa, tb, cb.dl, sc,
                                                              cnt.act_moves, c);
                if (tid == 0) {
                    sc.red[par][0] = sw;
                    sc.red[par][1] = c ? 1 : 0;
                }
                __syncthreads();
                sw = sc.red[par][0];
                conv = sc.red[par][1] != 0;
                par ^= 1;
                cnt.act_sweeps += sw;
                exact = false;                            // coordinates may have reached zero
            }
            // Working set: with the support converged, one scan of every
            // coordinate finds those that a sweep with the support held
            // would move.  None: that sweep would move nothing
            // (max |delta| = 0), so the lasso at this lambda is solved.
            // Otherwise, while their union with the support fits the phase
            // and one of them would move by tol or more, they join the next
            // phase's coordinates at b = 0, instead of the sweep moving them
            // one at a time with an O(p) update each.  Else the sweep decides.
            // After a phase the scan runs inside the gradient refresh.
            const bool ws = conv && rounds < BLK_WS_ROUNDS;
            bool scanned = false;
            int nv = 0;
            float mv = 0.f;
            // a handed-over support (at most LAZY_CAP entries) fits the list
            if (phase || stale) {
                if (uni) {                                // the support of the union
                    n = nl = block_filter_list<T>(b, ubuf, np, list, sc, par);
                    exact = true;
                }
                scanned = ws && n <= BLK_AMAX;
                const bool keep = scanned && bounds;      // what the scan leaves bounds for
                if (!scanned) cb.valid = false;
                gfull = !cb.valid;
                block_form_gradient<T, STD>(j, g, b, list, n, a, scanned, lam, sc,
                                            RefreshScan{vlist, BLK_AMAX, wp}, keep ? &cb : nullptr,
                                            plist, phase ? np : 0);
                __syncthreads();
                if (keep) {
                    // by warp 0, which is also the one that changes the list
                    if (tid < 32)
                        for (int e = tid; e < n; e += 32) cb.prev[e] = list[e];
                    cb.nprev = n;
                    cb.valid = true;
                }
                if (scanned) {
                    nv = sc.wcnt[wp];
                    mv = __int_as_float(sc.wmax[wp]);
                    wp ^= 1;
                }
                stale = false;
            }
            uni = false;
            if (ws && n <= BLK_AMAX) {
                if (!scanned) {
                    if (!gfull) form_all();
                    // no refresh (b = 0, g = S_.j): a scan of its own, the union into ubuf
                    nu = block_scan_list<T, STD>(j, g, b, a, lam, ubuf, sc, par, nv, mv);
                }
                ++cnt.sweeps;
                if (nv == 0) {
                    inner_ok = true;
                    break;
                }
                if (scanned) nu = n + nv;
                if (nu <= BLK_AMAX && (double)mv >= a.tol) {
                    if (scanned && tid < 32) warp_union(list, n, vlist, nv, ubuf);
                    __syncthreads();
                    uni = true;
                    ++rounds;
                    continue;
                }
            }
            if (!gfull) form_all();
            const T md = block_sweep<T, STD>(j, g, b, a, lam, conv, cand, cnt.moves, sc, par,
                                             (int)(cnt.sweeps - sweeps0));
            nl = -1;
            cb.valid = false;                             // the candidates have overwritten them
            ++cnt.sweeps;
            if ((double)md < a.tol) {
                inner_ok = true;
                break;
            }
        }
        if (!inner_ok) status |= COL_NOT_CONVERGED;
        const int n = support();
        double q;
        if (!block_quadratic_form_saa<T>(j, b, n, saa_list, saa_n, saa, a, sc, q))
            q = block_quadratic_form<T>(j, b, list, n, a, sc);
        if (tid < 32) {                                   // one warp on the FP64 pipe
            int f = (status & COL_DEGENERATE) ? 1 : 0;
            if (!(q > floor2)) {
                q = floor2;
                f = 1;
            }
            double sn = sqrt_heron(q);
            if (fabs(sn - sigma) < a.tol) f |= 2;
            if ((f & 2) || r + 1 == a.maxit) {            // this sigma is returned
                sn = sqrt_last(q, sn);
                if (tid == 0 && a.hand) a.hand[2 * (size_t)j + 1] = q;
            }
            double nxt = sn;
            if (r > 0 && r + 1 < a.maxit && !f)
                nxt = sigma_step(s_prev, (float)(f_prev - s_prev), sigma, sn, (float)(sn - sigma));
            if (tid == 0) {
                sc.sig[0] = sn;
                sc.sig[1] = nxt;
                sc.sigf = f;
            }
        }
        __syncthreads();
        const double sn = sc.sig[0], nxt = sc.sig[1];
        if (sc.sigf & 1) status |= COL_DEGENERATE;
        if (sc.sigf & 2) {
            sigma = sn;
            break;
        }
        s_prev = sigma;
        f_prev = sn;
        sigma = nxt;
    }
    if (r == a.maxit) {
        r = a.maxit - 1;
        status |= COL_NOT_CONVERGED;
    }
    // b_j into row j of BT (a list where it fits, see coef_cap), row j of Theta cleared
    T* brow = a.BT + (size_t)j * ldp;
    const int nb = support();
    if (nb <= coef_cap(ldp)) {
        int* idx = coef_idx(brow, ldp);
        for (int t = tid; t < nb; t += BLK_THREADS) {
            brow[t] = b[list[t]];
            idx[t] = list[t];
        }
    } else {
        for (int k = tid; k < ldp; k += BLK_THREADS) brow[k] = b[k];
    }
    if (a.Theta) clear_theta_row(a.Theta, a.p, j, tid, BLK_THREADS);
    if (tid == 0) a.nsup[j] = nb <= coef_cap(ldp) ? nb : -1;
    if (tid == 0) {
        a.sigma[j] = sigma;
        a.col_status[j] = status;
    }
    cnt.outer_max = max(cnt.outer_max, r + 1);
    cnt.max_sw = max(cnt.max_sw, (int)(cnt.sweeps - sweeps0));
    cnt.n_nc += (status & COL_NOT_CONVERGED) != 0;
    cnt.n_deg += (status & COL_DEGENERATE) != 0;
    ++cnt.blk;
    __syncthreads();
}

__device__ __forceinline__ void flush_counters_block(FitCtrl* ctrl, ColCounters& c) {
    if (threadIdx.x == 0) {
        if (c.blk) atomicAdd(&ctrl->block_cols, c.blk);
        if (c.sweeps) atomicAdd(&ctrl->total_sweeps, c.sweeps);
        if (c.moves) atomicAdd(&ctrl->moves, c.moves);
        if (c.act_sweeps) atomicAdd(&ctrl->act_sweeps, c.act_sweeps);
        if (c.act_moves) atomicAdd(&ctrl->act_moves, c.act_moves);
        atomicMax(&ctrl->outer_max, c.outer_max);
        atomicMax(&ctrl->max_col_sweeps, c.max_sw);
        if (c.n_nc) atomicAdd(&ctrl->n_not_converged, c.n_nc);
        if (c.n_deg) atomicAdd(&ctrl->n_degenerate, c.n_deg);
    }
    c = ColCounters();
}

// The nonzero entries of Theta of column j and its sigma in the original scale,
// by THETA_LANES lanes (Eq. (4), Eq. (9), Proposition 1; the arithmetic of
// theta_pair below).  Every pair with a coefficient in both lists is written to
// both mirrored entries by its smaller index.  The rows are clear (the solvers'
// clear_theta_row).  inv(k) is 1 / sigma_k^2 on the working scale.
// Dense rows of B^T and of Theta cost 0.52 GB written by the solvers, 0.55 GB
// read and 1.09 GB written in a pass of its own on the 256-fit batch, 0.373 ms
// after the descent; the scattered entries take 0.048 ms, and the clearing runs
// under the descent, which leaves DRAM idle (1.40 -> 1.48 ms).
constexpr int THETA_LANES = 8;
template <typename T, class Inv>
__device__ __forceinline__ unsigned theta_column(const T* __restrict__ BT,
                                                 const int* __restrict__ nsup, int p, int ldp, int j,
                                                 const double* __restrict__ sigma,
                                                 const double* __restrict__ cs,
                                                 double* __restrict__ Theta,
                                                 double* __restrict__ sigma_out, Inv inv) {
    const int sub = threadIdx.x & (THETA_LANES - 1);
    const T* __restrict__ row = BT + (size_t)j * ldp;
    const int n = nsup[j];
    const double cj = cs[j], inv_j = inv(j);
    if (sub == 0) {
        Theta[(size_t)j * p + j] = inv_j * (cj * cj);
        sigma_out[j] = sigma[j] / cj;
    }
    auto pair = [&](int k, T bkj) {                    // k > j, bkj = b_kj != 0
        const T bjk = coef_of<T>(BT, nsup, ldp, k, j);
        if (bjk == T(0)) return;
        const double ojk = -(double)bjk * inv(k);      // Omega_1[j][k]
        const double okj = -(double)bkj * inv_j;       // Omega_1[k][j]
        const double out = (fabs(ojk) > fabs(okj) ? okj : ojk) * (cj * cs[k]);
        Theta[(size_t)j * p + k] = out;
        Theta[(size_t)k * p + j] = out;
    };
    if (n >= 0) {
        const int* __restrict__ idx = coef_idx(row, ldp);
        for (int e = sub; e < n; e += THETA_LANES) {
            const int k = idx[e];
            if (k > j) pair(k, row[e]);
        }
        return sub == 0 ? (unsigned)n : 0u;
    }
    unsigned nnz = 0;
    for (int k = sub; k < p; k += THETA_LANES) {
        const T b = row[k];
        if (b != T(0)) {
            ++nnz;
            if (k > j) pair(k, b);
        }
    }
    return nnz;
}

// Theta from dense rows of B^T (the joint rule, the eager and the residual
// form), over pairs of TS x TS tiles: the
// tile of rows j0.., columns k0.. (j0 <= k0) and its mirror.  Omega_1 = -B D
// on the working scale, min-magnitude symmetrisation (for j < k a tie keeps
// omega_jk) and Omega^o = C Omega C.  Both coefficient tiles are read once
// into shared memory, and every entry of both Theta tiles is written, both
// entries of a pair with the same value, so Theta is exactly symmetric and
// needs no clearing beforehand.  Blocks of the first
// tile row also write sigma in the original scale; nonzero coefficients are
// counted into ctrl->nnz.  Block shape 32 x 8.  TS = 64 for FP32
// coefficients, 32 for FP64 (static shared memory).
template <typename T>
__host__ __device__ constexpr int theta_ts() { return sizeof(T) == 4 ? 64 : 32; }

// Tile pairs of a p x p Theta.
template <typename T>
__host__ __device__ inline int theta_pairs(int p) {
    const int t = (p + theta_ts<T>() - 1) / theta_ts<T>();
    return t * (t + 1) / 2;
}

template <typename T>
__device__ void theta_pair(const T* __restrict__ BT, int p, int ldp,
                           const double* __restrict__ sigma, const double* __restrict__ cs,
                           double* __restrict__ Theta, double* __restrict__ sigma_out,
                           FitCtrl* ctrl, int pair) {
    constexpr int TS = theta_ts<T>();
    __shared__ T tA[TS][TS + 1];    // tA[kk][jj] = BT[k0+kk][j0+jj] = b_jk
    __shared__ T tB[TS][TS + 1];    // tB[jj][kk] = BT[j0+jj][k0+kk] = b_kj
    // 1/sigma^2 and c for the pair's rows and columns: FP64 divisions are
    // expensive on this part, so each block does 2 TS of them
    __shared__ double inv_j[TS], inv_k[TS], c_j[TS], c_k[TS];
    const int t = (p + TS - 1) / TS;
    int a = 0, rem = pair;
    while (rem >= t - a) {
        rem -= t - a;
        ++a;
    }
    const int j0 = a * TS, k0 = (a + rem) * TS;
    const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
    const int lin = ty * 32 + tx;
    if (lin < 2 * TS) {
        const bool col = lin < TS;
        const int i = col ? k0 + lin : j0 + lin - TS;
        double inv = 0.0, c = 0.0;
        if (i < p) {
            const double s = sigma[i];
            inv = 1.0 / (s * s);
            c = cs[i];
        }
        if (col) { inv_k[lin] = inv; c_k[lin] = c; }
        else { inv_j[lin - TS] = inv; c_j[lin - TS] = c; }
    }
    if constexpr (sizeof(T) == 4) {
        // 16-byte reads: 16 lanes per 64-float row; columns p..ldp-1 of B are
        // zero, quads past the padded row are not read
        const int q = 4 * (tx & 15);
        for (int r = 2 * ty + (tx >> 4); r < TS; r += 16) {
            float4 va = make_float4(0.f, 0.f, 0.f, 0.f), vb = va;
            if (k0 + r < p && j0 + q < ldp) va = *reinterpret_cast<const float4*>(BT + (size_t)(k0 + r) * ldp + j0 + q);
            if (j0 + r < p && k0 + q < ldp) vb = *reinterpret_cast<const float4*>(BT + (size_t)(j0 + r) * ldp + k0 + q);
            tA[r][q] = va.x; tA[r][q + 1] = va.y; tA[r][q + 2] = va.z; tA[r][q + 3] = va.w;
            tB[r][q] = vb.x; tB[r][q + 1] = vb.y; tB[r][q + 2] = vb.z; tB[r][q + 3] = vb.w;
        }
    } else {
        for (int r = ty; r < TS; r += 8)
            for (int q = tx; q < TS; q += 32) {
                tA[r][q] = (k0 + r < p && j0 + q < p) ? BT[(size_t)(k0 + r) * ldp + j0 + q] : T(0);
                tB[r][q] = (j0 + r < p && k0 + q < p) ? BT[(size_t)(j0 + r) * ldp + k0 + q] : T(0);
            }
    }
    __syncthreads();
    // Theta_jk for j = j0 + jj, k = k0 + kk
    auto value = [&](int jj, int kk) -> double {
        const int j = j0 + jj, k = k0 + kk;
        // the scale (c_j c_k) is formed before it multiplies, so the value
        // does not depend on which of the pair computes it
        if (j == k) return inv_k[kk] * (c_j[jj] * c_k[kk]);
        const T bjk = tA[kk][jj];      // coefficient of x_j in regression k
        const T bkj = tB[jj][kk];      // coefficient of x_k in regression j
        if (bjk == T(0) && bkj == T(0)) return 0.0;   // both candidates are zero
        const double ojk = -(double)bjk * inv_k[kk];  // Omega_1[j][k]
        const double okj = -(double)bkj * inv_j[jj];  // Omega_1[k][j]
        double out;
        if (j < k) out = fabs(ojk) > fabs(okj) ? okj : ojk;
        else out = fabs(okj) > fabs(ojk) ? ojk : okj;  // pair (k, j) with k < j
        return out * (c_j[jj] * c_k[kk]);
    };
    // Every entry of the tile and of its mirror is written (Theta needs no
    // clearing first), each row segment by consecutive lanes.  Both entries
    // of a pair come from the same value(jj, kk), so Theta is exactly
    // symmetric; a diagonal tile is its own mirror and is written once.
    unsigned long long nnz = 0;
    for (int jj = ty; jj < TS; jj += 8) {
        const int j = j0 + jj;
        if (j >= p) break;
        for (int kk = tx; kk < TS; kk += 32) {
            const int k = k0 + kk;
            if (k >= p) break;
            nnz += (j != k && tB[jj][kk] != T(0)) + (j0 != k0 && tA[kk][jj] != T(0));
            Theta[(size_t)j * p + k] = value(jj, kk);
        }
    }
    if (j0 != k0) {
        for (int kk = ty; kk < TS; kk += 8) {
            const int k = k0 + kk;
            if (k >= p) break;
            for (int jj = tx; jj < TS; jj += 32) {
                const int j = j0 + jj;
                if (j >= p) break;
                Theta[(size_t)k * p + j] = value(jj, kk);
            }
        }
    }
    if (j0 == 0 && lin < TS && k0 + lin < p) sigma_out[k0 + lin] = sigma[k0 + lin] / cs[k0 + lin];
    // one atomic per warp
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nnz += __shfl_xor_sync(FULL_MASK, nnz, o);
    if (tx == 0 && nnz) atomicAdd(&ctrl->nnz, nnz);
}

}  // namespace spmesl
