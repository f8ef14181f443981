#pragma once
// Gram tile on the CUDA cores (FP32), shared by the single-fit and the batched
// Gram kernels.
//
// X is row-major n x p, so the k-th slice X[i, m0 .. m0+BM-1] of both operand
// tiles is a contiguous row segment: every global load is coalesced.  A tile
// (tm, tn) with tm <= tn writes itself and its mirror, so both triangles of S
// are stored with row-contiguous writes.  Column centring (Section 2.2)
// subtracts the column means on the way into shared memory.  Every entry is
// one FP32 chain of fused multiply-adds in sample order whatever the tile.
//
// Bound by the FP32 pipe.  Each thread keeps TM x TN entries and takes two of
// them per packed fused multiply-add (two roundings, as two single ones), so
// the shared-memory reads and the address arithmetic fit beside the products;
// the next BK samples are read into registers under the products of these.
// 128 x 128 tiles of 128 threads with 8 x 16 entries carry the large fits:
// p = 10000, n = 500 894 us, 56 TFLOP/s (8 x 8 entries: 991; with single
// multiply-adds 1300; 64 x 64 tiles with 4 x 4 entries 1715), p = 5000, n = 1000
// 498 us (874).  Below GRAM_WIDE_TILES of them, whose last wave is then a large
// part, 64 x 64 tiles of 128 threads with 8 x 4 entries are faster: p = 2500,
// n = 200 (210 wide tiles) 38.9 against 45.1 us, p = 2000 (136) 26.8 against
// 28.7 (49.1 before); p = 3000 (300) 49.3 against 45.1, p = 10000, n = 500 1006
// against 894.
#include <cuda_runtime.h>

#include "common.cuh"

namespace spmesl {

constexpr int GRAM_BM = 64;             // tile of small fits and batches
constexpr int GRAM_THREADS = 128;
constexpr int GRAM_WIDE = 128;          // tile of large fits
constexpr int GRAM_WIDE_THREADS = 128;
constexpr int GRAM_WIDE_TILES = 250;    // 128 x 128 tiles from which they are taken (152 SMs, two a
                                        // SM: four fifths of a wave)
constexpr int GRAM_BK = 16;             // rows of X per stage
constexpr int GRAM_WIDE_BK = 8;         // (the prefetch shares the registers with 128 entries)

// d = a * b + d on both halves, each rounded as one fused multiply-add.
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a,
                                     unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// VEC: the rows of X start on 16-byte boundaries and p is a multiple of 4, so a
// thread stages four columns of a sample with one 16-byte load and store.
template <int BM, int BK, int THREADS, int TM, int TN, bool VEC>
__device__ __forceinline__ void gram_tile(const float* __restrict__ X, int n, int p, int ldx,
                                          const float* __restrict__ mu, float* __restrict__ S,
                                          int lds, float inv_n, int tm, int tn) {
    constexpr int TX = BM / TN, TY = BM / TM;            // threads across and down the tile
    static_assert(TX * TY == THREADS && TM % 4 == 0 && TN % 4 == 0, "tile shape");
    constexpr int PER = BK * BM / THREADS;               // operand values a thread stages
    static_assert(THREADS % BM == 0 || BM % THREADS == 0, "staging");
    constexpr int MC = BM / 4;                           // mirror: columns staged at a time
    constexpr int OPS = 2 * 2 * BK * BM, OUT = MC * (BM + 1);
    __shared__ __align__(16) float raw[OPS > OUT ? OPS : OUT];
    float (*As)[BK][BM] = reinterpret_cast<float (*)[BK][BM]>(raw);
    float (*Bs)[BK][BM] = reinterpret_cast<float (*)[BK][BM]>(raw + 2 * BK * BM);
    const int tid = threadIdx.x;
    // a warp covers 8 threads across and 4 down, so that one operand read of the
    // warp is at most 128 distinct bytes
    static_assert(TX % 8 == 0 && TY % 4 == 0, "warp shape");
    const int warp = tid >> 5, lane = tid & 31;
    const int tx = warp % (TX / 8) * 8 + (lane & 7), ty = warp / (TX / 8) * 4 + (lane >> 3);
    const int m0 = tm * BM, n0 = tn * BM;

    unsigned long long acc[TM][TN / 2];
#pragma unroll
    for (int u = 0; u < TM; ++u)
#pragma unroll
        for (int v = 0; v < TN / 2; ++v) acc[u][v] = 0ull;

    float pa[PER], pb[PER];
    // value (q, t) of the thread's share: row e / BM of the stage, column e % BM
    auto fetch = [&](int i0) {
        if constexpr (VEC) {
#pragma unroll
            for (int q = 0; q < PER / 4; ++q) {
                const int e = 4 * (tid + q * THREADS);
                const int i = i0 + e / BM, ca = m0 + e % BM, cb = n0 + e % BM;
                float4 va = make_float4(0.f, 0.f, 0.f, 0.f), vb = va;
                if (i < n) {
                    const float* __restrict__ row = X + (size_t)i * ldx;
                    if (ca < p) va = *reinterpret_cast<const float4*>(row + ca);
                    if (cb < p) vb = *reinterpret_cast<const float4*>(row + cb);
                    if (mu) {
                        if (ca < p) { va.x -= mu[ca]; va.y -= mu[ca + 1]; va.z -= mu[ca + 2]; va.w -= mu[ca + 3]; }
                        if (cb < p) { vb.x -= mu[cb]; vb.y -= mu[cb + 1]; vb.z -= mu[cb + 2]; vb.w -= mu[cb + 3]; }
                    }
                }
                *reinterpret_cast<float4*>(pa + 4 * q) = va;
                *reinterpret_cast<float4*>(pb + 4 * q) = vb;
            }
        } else {
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int e = tid + q * THREADS;
                const int i = i0 + e / BM, ca = m0 + e % BM, cb = n0 + e % BM;
                pa[q] = pb[q] = 0.f;
                if (i < n) {
                    if (ca < p) pa[q] = X[(size_t)i * ldx + ca] - (mu ? mu[ca] : 0.f);
                    if (cb < p) pb[q] = X[(size_t)i * ldx + cb] - (mu ? mu[cb] : 0.f);
                }
            }
        }
    };
    auto stage = [&](int buf) {
        if constexpr (VEC) {
#pragma unroll
            for (int q = 0; q < PER / 4; ++q) {
                const int e = 4 * (tid + q * THREADS);
                *reinterpret_cast<float4*>(&As[buf][e / BM][e % BM]) = *reinterpret_cast<float4*>(pa + 4 * q);
                *reinterpret_cast<float4*>(&Bs[buf][e / BM][e % BM]) = *reinterpret_cast<float4*>(pb + 4 * q);
            }
        } else {
#pragma unroll
            for (int q = 0; q < PER; ++q) {
                const int e = tid + q * THREADS;
                As[buf][e / BM][e % BM] = pa[q];
                Bs[buf][e / BM][e % BM] = pb[q];
            }
        }
    };
    fetch(0);
    stage(0);
    __syncthreads();
    int buf = 0;
    for (int i0 = 0; i0 < n; i0 += BK, buf ^= 1) {
        const bool more = i0 + BK < n;
        if (more) fetch(i0 + BK);
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            float a[TM];
            unsigned long long b[TN / 2];
#pragma unroll
            for (int g = 0; g < TM / 4; ++g)
                *reinterpret_cast<float4*>(a + 4 * g) =
                    *reinterpret_cast<const float4*>(&As[buf][kk][g * 4 * TY + 4 * ty]);
#pragma unroll
            for (int g = 0; g < TN / 4; ++g) {
                const ulonglong2 q =
                    *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][g * 4 * TX + 4 * tx]);
                b[2 * g] = q.x;
                b[2 * g + 1] = q.y;
            }
#pragma unroll
            for (int u = 0; u < TM; ++u) {
                const unsigned long long aa = pack2(a[u], a[u]);
#pragma unroll
                for (int v = 0; v < TN / 2; ++v) fma2(acc[u][v], aa, b[v]);
            }
        }
        if (more) stage(buf ^ 1);
        __syncthreads();
    }
    float out[TM][TN];
#pragma unroll
    for (int u = 0; u < TM; ++u)
#pragma unroll
        for (int v = 0; v < TN / 2; ++v) {
            unpack2(acc[u][v], out[u][2 * v], out[u][2 * v + 1]);
            out[u][2 * v] *= inv_n;
            out[u][2 * v + 1] *= inv_n;
        }
    const bool vec = (lds & 3) == 0 && (reinterpret_cast<uintptr_t>(S) & 15) == 0;
#pragma unroll
    for (int u = 0; u < TM; ++u) {
        const int r = m0 + (u / 4) * 4 * TY + 4 * ty + u % 4;
        if (r >= p) continue;
#pragma unroll
        for (int g = 0; g < TN / 4; ++g) {
            const int c = n0 + g * 4 * TX + 4 * tx;
            float* __restrict__ dst = S + (size_t)r * lds + c;
            if (vec && c + 3 < p) {
                *reinterpret_cast<float4*>(dst) = make_float4(out[u][4 * g], out[u][4 * g + 1],
                                                              out[u][4 * g + 2], out[u][4 * g + 3]);
            } else {
#pragma unroll
                for (int v = 0; v < 4; ++v)
                    if (c + v < p) dst[v] = out[u][4 * g + v];
            }
        }
    }
    if (tm != tn) {
        // the mirror, MC columns at a time through shared memory (the operands'
        // buffers: the loop above ended with a barrier)
        float (*Cs)[BM + 1] = reinterpret_cast<float (*)[BM + 1]>(raw);
        for (int cb = 0; cb < BM; cb += MC) {
#pragma unroll
            for (int g = 0; g < TN / 4; ++g) {
                const int c = g * 4 * TX + 4 * tx - cb;
                if (c >= 0 && c < MC) {
#pragma unroll
                    for (int v = 0; v < 4; ++v)
#pragma unroll
                        for (int u = 0; u < TM; ++u)
                            Cs[c + v][(u / 4) * 4 * TY + 4 * ty + u % 4] = out[u][4 * g + v];
                }
            }
            __syncthreads();
            for (int e = tid; e < MC * BM; e += THREADS) {
                const int c = e / BM, r = e % BM;
                if (n0 + cb + c < p && m0 + r < p)
                    S[(size_t)(n0 + cb + c) * lds + m0 + r] = Cs[c][r];
            }
            __syncthreads();
        }
    }
}

// Sum over the 8 sample groups of a 32 x 8 block (threadIdx.y) in a fixed order;
// valid in every thread of threadIdx.y = 0.
constexpr int MEAN_GROUPS = 8;
__device__ __forceinline__ double group_sum(double v, double (&part)[MEAN_GROUPS][33]) {
    part[threadIdx.y][threadIdx.x] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.y == 0) {
#pragma unroll
        for (int g = 0; g < MEAN_GROUPS; ++g) t += part[g][threadIdx.x];
    }
    __syncthreads();
    return t;
}

// Means of columns c0 .. c0 + 31 of X (for centring) by a 32 x 8 block, FP64
// accumulation: every eighth sample by one thread, the eight sums in turn.
// Bound by FP64 latency and by the FP64 pipes of the SMs that take part: one
// thread per column in blocks of 256 took 38 us at p = 1003, n = 251 (4 SMs,
// one chain of n additions), blocks of one warp 22, this 7.
template <typename T>
__device__ __forceinline__ void column_means(const T* __restrict__ X, int n, int p, int ldx,
                                             T* __restrict__ mu, int c0) {
    __shared__ double part[MEAN_GROUPS][33];
    const int c = c0 + threadIdx.x;
    double acc = 0.0;
    if (c < p) {
#pragma unroll 8
        for (int i = threadIdx.y; i < n; i += MEAN_GROUPS) acc += (double)X[(size_t)i * ldx + c];
    }
    acc = group_sum(acc, part);
    if (threadIdx.y == 0 && c < p) mu[c] = (T)(acc / n);
}

// Upper-triangular tile index -> (tm, tn), tm <= tn, for a t x t tile grid
// enumerated row by row: row tm holds t - tm tiles.
__device__ __forceinline__ void upper_tile(int idx, int t, int& tm, int& tn) {
    int row = 0, rem = idx;
    while (rem >= t - row) {
        rem -= t - row;
        ++row;
    }
    tm = row;
    tn = row + rem;
}

}  // namespace spmesl
