#pragma once
// FP64 Gram on the tensor cores: the pieces shared by the single-fit path
// (spmesl_gram with SPMESL_FP64) and the batched one (see gram_f64.cu).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <limits.h>

#include "gram_tc.cuh"

namespace spmesl {

constexpr int F64_SLICES = 7;         // 8-bit digits of a column's scaled values
constexpr int F64_LEVELS = 8;         // sums of digit products by weight (see gram_f64.cu)
constexpr int F64_SLAB = 4096;        // samples whose digits are held at a time
constexpr int F64_BN = 64;            // output tile: TC_BM rows x F64_BN columns
constexpr int F64_EXPO_DIRECT = INT_MAX;   // column whose products are formed directly in FP64
constexpr int F64_EXPO_MAX = 400;     // largest |exponent| that the digits' scaling handles

// Samples of a digit plane's row.  The planes take 14 bytes a sample, 1.75 times X:
// data of more than F64_SLAB samples go through them in slabs, with the sums of the
// digit products kept in S's lower triangle between two.
__host__ __device__ inline int f64_plane_n(int n) {
    return tc_pad_n(n) < F64_SLAB ? tc_pad_n(n) : F64_SLAB;
}
static_assert(F64_SLAB % TC_NPAD == 0, "slabs");

// One fit: TMA maps over its digit planes D ([F64_SLICES][p][f64_plane_n] bf16; boxes
// of 128 and 64 columns of X), the columns' exponents, the data and the output.
struct F64Fit {
    CUtensorMap ma, mb;
    const double* X;
    const double* mu;
    const int* expo;
    const int* marks;     // per 32 columns whether one of them is F64_EXPO_DIRECT
    double* S;
    int n, p, ldx, lds, tile_start;
    double inv_n;
    TileGrid g;
};

// The fits of one launch: device table, tile_start ascending, the fit of each tile,
// and the marks of all fits in one array.
struct F64Batch {
    const F64Fit* fits;
    const int* tile_fit;
    const int* marks;
    int n_fits, n_tiles, n_marks;
    int n_blocks;         // sum of f64_direct_blocks
    int s0;               // first sample of the slab
};

// The counts behind the exponents.
__host__ __device__ inline unsigned* f64_counts(int* expo, int p) {
    return reinterpret_cast<unsigned*>(expo + p + (p + 31) / 32);
}

// Bytes of the digit planes, and of the exponents followed by the marks and, per column,
// the two counts of the rule on small samples (256-byte aligned each).
inline size_t f64_digit_bytes(int n, int p) {
    return align_up((size_t)F64_SLICES * p * f64_plane_n(n) * 2, 256);
}
inline size_t f64_expo_bytes(int p) { return align_up((3 * (size_t)p + (p + 31) / 32) * 4, 256); }
int f64_direct_blocks(int p);

// x as an integer v = round(x 2^(55 - E)) for |x| < 2^E, and its balanced
// base-256 digits: v = sum_s d[s] 256^(6 - s), |d[s]| <= 128.
__device__ __forceinline__ void f64_digits(double x, int E, int (&d)[F64_SLICES]) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x);
    const int e = (int)(u >> 52) & 0x7ff;
    unsigned long long m = u & 0xfffffffffffffull;
    if (e) m |= 1ull << 52;
    const int sh = max(e, 1) - 1020 - E;            // at most 2
    unsigned long long a;
    if (sh >= 0) a = m << sh;
    else a = sh < -54 ? 0ull : (m + (1ull << (-sh - 1))) >> -sh;
    long long v = (u >> 63) ? -(long long)a : (long long)a;
#pragma unroll
    for (int s = F64_SLICES - 1; s > 0; --s) {
        d[s] = (int)(signed char)(v & 255);          // balanced remainder in [-128, 127]
        v = (v - d[s]) >> 8;
    }
    d[0] = (int)v;
}

// Whether x counts for F64_EXPO_DIRECT's rule: 1 for a nonzero value, and 2^16
// more when it is below 2^(E - F64_SMALL).
constexpr int F64_SMALL = 10;
__device__ __forceinline__ unsigned f64_small(double x, int E) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x) << 1;
    const int e = (int)(u >> 53);                     // |x| in [2^(e - 1023), 2^(e - 1022))
    return u == 0ull ? 0u : (e - 1022 <= E - F64_SMALL ? 0x10001u : 1u);
}

// Exponents and digit planes of columns c0 .. c0 + 31 of X, centred by mu when
// given (block 32 x 8), and the block's mark.  The largest magnitude of a column sets its exponent
// E (|x| < 2^E); a column with a non-finite value or an exponent beyond
// F64_EXPO_MAX is marked F64_EXPO_DIRECT and gets zero digits.  So is, by its
// digits' own pass, a column with more than a quarter of its nonzero samples
// below 2^(E - F64_SMALL): a few samples that large set the digits' unit, and an FP64
// sum in which they meet small partners is closer than the digits are.  Normal samples
// pass the rule by far (0.5 % of them are that small), Student t with 2 degrees too;
// log-normal (s = 3) and Cauchy columns and a column of ordinary samples with one of
// 10^3 or more are marked.  Magnitudes are
// compared and digits formed on the integer pipe: the FP64 pipe takes 16 cycles
// an instruction.  Samples from n to the next multiple of 64 are written as zeros.  Each pass of 64
// samples loads the next one's (81 -> 78 us for 50 fits of p = 500, n = 250).
// One slab of samples a call, s0 its first; the first one forms the exponents of all, the
// last one the marks.
__device__ __forceinline__ void f64_digit_columns(const double* __restrict__ X, int n, int p,
                                                  int ldx, const double* __restrict__ mu,
                                                  int* __restrict__ expo, int* __restrict__ mark,
                                                  unsigned* __restrict__ counts,
                                                  __nv_bfloat16* __restrict__ D, int c0, int s0) {
    __shared__ long long red[8][33];
    __shared__ int sE[32];
    __shared__ unsigned nonzero[32], small[32];        // samples of each column (by its warp)
    __shared__ double tile[32][65];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int cl = c0 + tx;
    const double m = (mu && cl < p) ? mu[cl] : 0.0;
    long long mx = 0;
    if (cl < p && s0 == 0) {
#pragma unroll 8
        for (int i = ty; i < n; i += 8) {
            double v = X[(size_t)i * ldx + cl];
            if (mu) v -= m;
            mx = max(mx, __double_as_longlong(v) & 0x7fffffffffffffffll);
        }
    }
    red[ty][tx] = mx;
    __syncthreads();
    if (ty == 0) {
#pragma unroll
        for (int r = 1; r < 8; ++r) mx = max(mx, red[r][tx]);
        const int e = (int)(mx >> 52);
        int E = mx == 0 ? 0 : e - 1022;
        if (e == 0x7ff || E > F64_EXPO_MAX || E < -F64_EXPO_MAX) E = F64_EXPO_DIRECT;
        if (s0 != 0) E = cl < p ? expo[cl] : 0;
        sE[tx] = E;
        nonzero[tx] = small[tx] = 0u;
        if (cl < p) expo[cl] = E;
    }
    __syncthreads();
    const int ldd = f64_plane_n(n), end = s0 + min(tc_pad_n(n) - s0, F64_SLAB);
    const size_t plane = (size_t)p * ldd;
    double nx[8];                         // the next 64 samples, on their way during the digits
    auto fetch = [&](int i0) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int i = i0 + ty + 8 * r;
            nx[r] = (i < n && cl < p) ? X[(size_t)i * ldx + cl] : m;
        }
    };
    fetch(s0);
    for (int i0 = s0; i0 < end; i0 += 64) {
#pragma unroll
        for (int r = 0; r < 8; ++r) tile[tx][ty + 8 * r] = mu ? nx[r] - m : nx[r];
        __syncthreads();
        if (i0 + 64 < end) fetch(i0 + 64);
        for (int r = ty; r < 32; r += 8) {
            const int c = c0 + r;
            if (c < p) {
                const int E = sE[r];
                int d0[F64_SLICES], d1[F64_SLICES];
                if (E == F64_EXPO_DIRECT) {
#pragma unroll
                    for (int s = 0; s < F64_SLICES; ++s) d0[s] = d1[s] = 0;
                } else {
                    const double x0 = tile[r][2 * tx], x1 = tile[r][2 * tx + 1];
                    f64_digits(x0, E, d0);
                    f64_digits(x1, E, d1);
                    const unsigned few = __reduce_add_sync(FULL_MASK, f64_small(x0, E) + f64_small(x1, E));
                    if (tx == 0) {
                        nonzero[r] += few & 0xffffu;
                        small[r] += few >> 16;
                    }
                }
                __nv_bfloat16* out = D + (size_t)c * ldd + (i0 - s0) + 2 * tx;
#pragma unroll
                for (int s = 0; s < F64_SLICES; ++s) {
                    // |d| <= 128 is exact in bf16: the upper half of its FP32 bits
                    // (made FP32 by the 1.5 2^23 offset, off the conversion pipe)
                    const float f0 = __int_as_float(0x4b400000 + d0[s]) - 12582912.0f;
                    const float f1 = __int_as_float(0x4b400000 + d1[s]) - 12582912.0f;
                    *reinterpret_cast<unsigned*>(out + s * plane) =
                        __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
                }
            }
        }
        __syncthreads();
    }
    bool direct = false;                  // (lane 0) a column of this warp
    if (tx == 0) {
        for (int r = ty; r < 32; r += 8) {
            if (c0 + r >= p) continue;
            if (s0 != 0) {
                nonzero[r] += counts[2 * (c0 + r)];
                small[r] += counts[2 * (c0 + r) + 1];
            }
            if (end < n) {
                counts[2 * (c0 + r)] = nonzero[r];
                counts[2 * (c0 + r) + 1] = small[r];
                continue;
            }
            const bool few = 4ull * small[r] > nonzero[r];
            if (few) expo[c0 + r] = F64_EXPO_DIRECT;
            direct |= few || sE[r] == F64_EXPO_DIRECT;
        }
    }
    direct = __syncthreads_or(direct);
    if (tx == 0 && ty == 0) *mark = direct ? 1 : 0;
}

// Fill f (host side).  False if the tensor maps could not be encoded.
bool f64_encode_fit(F64Fit& f, const double* X, int n, int p, int ldx, const double* mu,
                    const int* expo, const int* marks, const void* D, double* S, int lds,
                    int tile_start);

// One persistent launch over the tiles of a batch (as launch_gram_tc_batch).
cudaError_t launch_gram_f64_batch(const F64Batch& b, cudaStream_t st);

}  // namespace spmesl
