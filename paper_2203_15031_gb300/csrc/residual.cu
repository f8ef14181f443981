// Coordinate descent for SPMESL in the residual form, without the Gram
// matrix (sm_103a).  Algorithm 3 keeps the residual matrix E = X - X B and
// forms each coordinate's gradient from the data (a_kj = x_k' e_j / n), and
// Proposition 2 updates E by a rank-1 term after every move; this file runs
// that form per column, with the cyclic ascending order and the per-column
// stopping rule of Algorithm 1.
//
// Layout in HBM (see res_layout):
//   W   ldn x ldp  W[i][k] = w_k[i], the scaled data, rows past n and columns
//                  past p zero
//   Wt  p x ldn    Wt[k][i] = w_k[i] (the same values, transposed)
//   BT  p x ldp    row j = coefficients b_.j of regression j
// with w_k = (x_k - mu_k) c_k / sqrt(n), c_k = s_kk^-1/2 when standardising
// (else 1), so that w_k' w_l = S^C_kl: the working matrix of the covariance
// form is never formed.  Memory is O(n p) for the data plus the p x p
// coefficients; the covariance form needs three p x p matrices besides S.
//
// One warp solves one column j at a time and keeps its residual
// r_j = w_j - W b_j (n values) in shared memory, with the sorted support of
// b_j and per-chunk summaries.  The gradient of coordinate k is
// g_kj = w_k' r_j, the same quantity S^C_kj - S^C_k. b_j that the covariance
// form keeps.  A sweep walks 128-coordinate chunks: the chunk's slice of g_j
// is W[:, chunk]' r_j (n coalesced 512-byte row reads, r_j broadcast from
// shared memory), the first coordinate that moves is found by ballot, its
// move updates r_j -= w_k delta from row k of Wt, and the slice is formed
// again from the new r_j.  sigma_j^2 = ||r_j||^2 (Eq. (14)) is formed in FP64
// from a residual recomputed from the data, which also removes the rounding
// drift of the running r_j.  No active-set phase: the iterates are those of
// plain cyclic sweeps (Algorithm 1).
//
// What bounds it: the longest column's chain of slices and moves (one warp).
// Chunks whose coordinates at zero provably stay there have only their support
// coordinates formed, one n-term dot each, over a row that the warp loads ahead;
// a slice is formed once, not after each of its moves.  Erdos-Renyi p = 2000,
// n = 200, FP32, a fit: 16.9 ms with a whole slice formed per visit and per move;
// 4.3 ms with quiet chunks; 3.5 ms with the growth bounded per chunk; 1.77 ms
// with rows staged through shared memory (a visit 3800 -> under 1000 cycles)
// and single coordinates formed after a move.  Testing a quiet chunk again after each of
// its moves takes 3.6 % of that fit.  The same iterates bit for bit.  Without standardisation
// there are no such bounds, and every move is followed by the chunk's slice.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>

#include "cd_device.cuh"
#include "gram_device.cuh"

namespace spmesl {
namespace {

constexpr int RES_MAX_N = 16384;   // the skip margins below assume n <= 2^14

template <typename T>
struct ResArgs {
    const T* W;
    const T* Wt;
    T* BT;
    const T* diag;       // ||w_k||^2 (unstandardised update)
    const unsigned char *cmax0, *cmax1;   // bounds of |w_k' w_l| (see chunk_bound)
    int cm_chunks;       // 128-coordinate chunks per byte of them
    int stage;           // 1: support rows go through shared memory (n <= RES_ROW * 32)
    double* sigma;       // working-scale sigma
    int* col_status;
    FitCtrl* ctrl;
    int n, ldn, p, ldp, maxit;
    double lambda0, tol;
};

// A bound of |w_k' w_l| over the coordinates l != k of chunk c (standardised
// data): sixteen bytes per column, each for cm_chunks chunks (one up to
// p = 2048), in units of 1/254.  They take the place of the column means and
// scales once the scaled data are built, so the workspace is O(n p) as before.
constexpr int CM_GROUPS = 16;
template <typename T>
__device__ __forceinline__ float chunk_bound(const ResArgs<T>& a, int k, int c) {
    const int g = a.cm_chunks == 1 ? c : c / a.cm_chunks;
    const unsigned char* t = g < 8 ? a.cmax0 + g : a.cmax1 + (g - 8);
    return (float)t[8 * (size_t)k] * ((1.0f + 0x1p-20f) / 254.0f);
}

// Samples of a support row that the warp holds in registers (32 per register).
constexpr int RES_ROW = 16;
// Coordinates of a chunk that are formed one by one after a move.
constexpr int RES_OPEN = 12;

// Upper bounds on ||r_j|| (warp-uniform): rb now, rmax over the solve so far.
struct ResNorm {
    float rb, rmax;
};

template <typename T>
__host__ __device__ constexpr size_t res_warp_smem_bytes(int ldn, int ldp) {
    return (size_t)ldn * sizeof(T) + (size_t)LAZY_CAP * (sizeof(int) + sizeof(T)) +
           (size_t)num_chunks(ldp) * sizeof(ChunkInfo);
}

template <typename T>
__device__ __forceinline__ void lds4(const T* __restrict__ src, T (&v)[4]) {
    if constexpr (sizeof(T) == 4) {
        const float4 q = *reinterpret_cast<const float4*>(src);
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    } else {
        const double2 q0 = *reinterpret_cast<const double2*>(src);
        const double2 q1 = *reinterpret_cast<const double2*>(src + 2);
        v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
    }
}

// acc[t] = sum_i W[i][k0 + t] r[i] over i < n4 (a multiple of 4; rows of W
// and entries of r past n are zero).  Two interleaved partial sums.  A slice
// is n 512-byte rows from L2, bound by the loads one warp has in flight:
// sixteen (p = 2000 columns leave only 13 warps an SM, so registers are free).
template <typename T>
__device__ __forceinline__ void slice_dot(const T* __restrict__ W, int ldp, int n4, int k0,
                                          const T* __restrict__ r, T (&acc)[SCAN_V]) {
    T a0[SCAN_V] = {T(0), T(0), T(0), T(0)}, a1[SCAN_V] = {T(0), T(0), T(0), T(0)};
    const T* w = W + k0;
#pragma unroll(sizeof(T) == 4 ? 4 : 2)
    for (int i = 0; i < n4; i += 4) {
        T rv[4];
        lds4<T>(r + i, rv);
        T z0[SCAN_V], z1[SCAN_V], z2[SCAN_V], z3[SCAN_V];
        load4g<T>(w + (size_t)i * ldp, z0);
        load4g<T>(w + (size_t)(i + 1) * ldp, z1);
        load4g<T>(w + (size_t)(i + 2) * ldp, z2);
        load4g<T>(w + (size_t)(i + 3) * ldp, z3);
#pragma unroll
        for (int t = 0; t < SCAN_V; ++t) {
            a0[t] = fma(z0[t], rv[0], a0[t]);
            a1[t] = fma(z1[t], rv[1], a1[t]);
            a0[t] = fma(z2[t], rv[2], a0[t]);
            a1[t] = fma(z3[t], rv[3], a1[t]);
        }
    }
#pragma unroll
    for (int t = 0; t < SCAN_V; ++t) acc[t] = a0[t] + a1[t];
}

// The same sum for one coordinate from its row of Wt (Wt[k][i] = W[i][k]):
// the products and their order are those of slice_dot, so the result is the
// value that the chunk's slice holds at coordinate k.  Every lane forms it
// (uniform reads of r and of the row, which is staged in shared memory).
template <typename T, bool SMEM>
__device__ __forceinline__ T column_dot(const T* __restrict__ wk, int n4, const T* __restrict__ r) {
    T a0 = T(0), a1 = T(0);
#pragma unroll(sizeof(T) == 4 ? 8 : 4)
    for (int i = 0; i < n4; i += 4) {
        T rv[4], z[4];
        lds4<T>(r + i, rv);
        if constexpr (SMEM) lds4<T>(wk + i, z);
        else load4g<T>(wk + i, z);
        a0 = fma(z[0], rv[0], a0);
        a1 = fma(z[1], rv[1], a1);
        a0 = fma(z[2], rv[2], a0);
        a1 = fma(z[3], rv[3], a1);
    }
    return a0 + a1;
}

// Row k of Wt in the warp's registers (entry lane + 32 i in v[i]; n <= RES_ROW * 32).
template <typename T>
__device__ __forceinline__ void load_row(const ResArgs<T>& a, int k, T (&v)[RES_ROW]) {
    const T* __restrict__ wk = a.Wt + (size_t)k * a.ldn + (threadIdx.x & 31);
#pragma unroll
    for (int i = 0; i < RES_ROW; ++i)
        if (32 * i < a.n) v[i] = __ldg(wk + 32 * i);
}

// The gradient of one coordinate k at the current residual: its row through the
// stage buffer (from registers when the caller has loaded it), or from global
// memory when n is beyond it.
template <typename T>
__device__ __forceinline__ T coordinate_dot(const ResArgs<T>& a, int k, const T (&v)[RES_ROW],
                                            T* __restrict__ stage, const T* __restrict__ r) {
    const int n4 = (a.n + 3) & ~3;
    if (!a.stage) return column_dot<T, false>(a.Wt + (size_t)k * a.ldn, n4, r);
    __syncwarp();                       // the last row's readers are done
#pragma unroll
    for (int i = 0; i < RES_ROW; ++i)
        if (32 * i < a.n) stage[32 * i + (threadIdx.x & 31)] = v[i];
    __syncwarp();
    return column_dot<T, true>(stage, n4, r);
}

// Per-chunk summary of the residual form: after the chunk was last scanned, the
// largest |g_k| over its coordinates with b_k = 0, a bound of how far any of them
// has moved since, the move count at that moment, and whether it holds support.
struct ResChunk {
    float maxabs, grow;
    unsigned moves_at;
    int nsupp;
};
static_assert(sizeof(ResChunk) == sizeof(ChunkInfo), "res_warp_smem_bytes counts ChunkInfo");

// Scan state of one column (warp-uniform).
struct ResScan {
    ResChunk* ci;
    unsigned nmoves;
};

// A chunk is quiet when none of its coordinates at zero can reach
// the threshold.  Since the chunk was scanned, each move delta_m changed the
// exact dot w_k' r by |delta_m w_k' w_m| <= |delta_m| cmax[m][chunk] (the bound
// is a quarter of the Cauchy-Schwarz one at p = 2000, n = 200, and most of a
// column's slices were formed for the difference), plus the rounding of the r
// update (2^-24 ||r||), and each residual
// recomputation was entered as a move of size ||r_new - r_old|| in every chunk; each of the
// two computed dots (then and now) is within n 2^-24 ||r|| of the exact one
// (Cauchy-Schwarz, ||w_k|| <= 1 + 2^-22).  With rmax bounding ||r|| over the
// solve, the margins below cover these terms, the rounding of the growth's
// sum (each of the dm additions is off by at most 2^-24 of it) and of the bound
// itself.  A coordinate at zero
// in a quiet chunk would therefore have computed |g_k| < lambda and not moved:
// a quiet chunk without support is skipped, and in one with support only the
// support coordinates are formed and tested, in their order, for as long as the
// chunk stays quiet under their moves; after a move that may have carried a
// coordinate at zero to the threshold the rest of the chunk is scanned.  So the sweep is
// the same as a full scan.  (maxabs covers the coordinates that were zero
// when the chunk was scanned; one that has come to zero since marks its chunk,
// maxabs = infinity.)
__device__ __forceinline__ bool quiet_chunk(const ResChunk& c, unsigned nmoves, float lam, float rmax,
                                            int n) {
    const unsigned dm = nmoves - c.moves_at;
    if (dm > 4096u) return false;
    const float bound = c.maxabs * (1.0f + 0x1p-22f) + c.grow * (1.0f + 0x1p-10f) +
                        c.grow * (float)(dm + 2u) * 0x1p-23f +
                        rmax * (float)(n + (int)dm + 2) * 0x1p-22f + lam * 0x1p-20f;
    return bound < lam;
}

// Chunks of [from, from + 32) that the sweep must visit (standardised data),
// and in `full` those of them whose slice must be formed (see quiet_chunk).
template <bool STD>
__device__ __forceinline__ unsigned res_chunks_to_visit(const ResScan& cs, int from, int nch,
                                                        float lam, float rmax, int n,
                                                        unsigned& full) {
    const int ci = from + (int)(threadIdx.x & 31);
    bool scan = ci < nch, visit = scan;
    if constexpr (STD) {
        if (scan) {
            const ResChunk c = cs.ci[ci];
            scan = !quiet_chunk(c, cs.nmoves, lam, rmax, n);
            visit = scan || c.nsupp != 0;
        }
    }
    full = __ballot_sync(FULL_MASK, scan);
    return __ballot_sync(FULL_MASK, visit);
}

// Whether a move's row goes through the warp's registers, loaded before the move is formed.
// Unstandardised FP64 fits gain nothing (p = 100, n = 50 4.54 ms with, 4.37 without),
// FP32 ones half their time (p = 2000, n = 200 6.2 against 10.3).
template <typename T, bool STD>
__device__ constexpr bool row_in_registers() { return STD || sizeof(T) == 4; }

// A move of coordinate k by delta: Proposition 2's r_j -= w_k delta (row k of
// Wt, in v with the stage buffer) and the chunks' growth.
template <typename T, bool STD>
__device__ __forceinline__ void note_residual_move(T* __restrict__ r, int k, const ResArgs<T>& a,
                                                   const T (&v)[RES_ROW], T delta, ResScan& cs,
                                                   ResNorm& rn) {
    const int n = a.n, lane = threadIdx.x & 31;
    ++cs.nmoves;
    if constexpr (STD) {
        const int nch = num_chunks(a.ldp);
        for (int c = lane; c < nch; c += 32)
            cs.ci[c].grow += fabsf((float)delta) * chunk_bound(a, k, c);
    }
    rn.rb = (rn.rb + fabsf((float)delta)) * (1.0f + 0x1p-19f);
    rn.rmax = fmaxf(rn.rmax, rn.rb);
    __syncwarp();                       // every lane has read r
    if (row_in_registers<T, STD>() && a.stage) {
#pragma unroll
        for (int i = 0; i < RES_ROW; ++i)
            if (32 * i + lane < n) r[32 * i + lane] = fma(-delta, v[i], r[32 * i + lane]);
    } else {
        const T* __restrict__ wk = a.Wt + (size_t)k * a.ldn;
        for (int i = lane; i < n; i += 32) r[i] = fma(-delta, wk[i], r[i]);
    }
    __syncwarp();
}

// One sweep over all coordinates of column j; returns max |delta b|.  Sets
// `overflow` and stops if the support list is full (the move is not applied).
template <typename T, bool STD>
__device__ T sweep_residual(int j, Support<T>& s, T* __restrict__ r, T* __restrict__ stage,
                            const ResArgs<T>& a, T lam,
                            unsigned long long& moves, ResScan& cs, ResNorm& rn, bool& overflow) {
    const int lane = threadIdx.x & 31;
    const int p = a.p, ldp = a.ldp;
    const int n4 = (a.n + 3) & ~3;
    const int nch = (p + CHUNK - 1) / CHUNK;
    T maxd = T(0);
    int e0 = 0;
    int mbase = 0;
    unsigned full;
    unsigned mask = res_chunks_to_visit<STD>(cs, 0, nch, (float)lam, rn.rmax, a.n, full);
    for (;;) {
        if (mask == 0u) {
            mbase += 32;
            if (mbase >= nch) break;
            mask = res_chunks_to_visit<STD>(cs, mbase, nch, (float)lam, rn.rmax, a.n, full);
            continue;
        }
        const int bit = __ffs(mask) - 1;
        const int ci = mbase + bit;
        mask &= mask - 1u;
        const int cb = ci * CHUNK;
        while (e0 < s.n && s.idx[e0] < cb) ++e0;
        int e1 = e0;
        while (e1 < s.n && s.idx[e1] < cb + CHUNK) ++e1;
        const unsigned nmoves0 = cs.nmoves;
        int cursor = cb;
        if constexpr (STD) {
            if (!((full >> bit) & 1u)) {
                // a quiet chunk: its support coordinates in turn.  One costs a
                // chain of n/2 fused multiply-adds over its row, which is loaded
                // under the chain before it; the whole slice it replaces read
                // n rows of 512 bytes from L2.
                T nx[RES_ROW];
                bool quiet = true;
                // of the coordinates that were zero when the chunk was visited: one that comes
                // to zero now is behind the sweep and opens the chunk for the next one
                const float maxabs = cs.ci[ci].maxabs;
                if (a.stage && e0 < e1) load_row<T>(a, s.idx[e0], nx);
                for (int e = e0; e < e1;) {
                    const int k = s.idx[e];
                    const T bk = s.val[e];
                    T v[RES_ROW];
#pragma unroll
                    for (int i = 0; i < RES_ROW; ++i) v[i] = nx[i];
                    if (a.stage && e + 1 < e1) load_row<T>(a, s.idx[e + 1], nx);
                    const T nb = soft<T>(coordinate_dot<T>(a, k, v, stage, r) + bk, lam);  // ||w_k||^2 = 1
                    if (nb == bk) {
                        ++e;
                        continue;
                    }
                    const T delta = nb - bk;
                    __syncwarp();                 // every lane has read the list
                    support_set<T>(s, e, k, nb);
                    if (nb == T(0)) {
                        --e1;
                        if (lane == 0) cs.ci[ci].maxabs = INFINITY;
                    } else {
                        ++e;
                    }
                    maxd = fmax(maxd, fabs(delta));
                    note_residual_move<T, STD>(r, k, a, v, delta, cs, rn);
                    ++moves;
                    ResChunk c = cs.ci[ci];
                    c.maxabs = maxabs;
                    if (!quiet_chunk(c, cs.nmoves, (float)lam, rn.rmax, a.n)) {
                        quiet = false;            // the coordinates after k are scanned
                        cursor = k + 1;
                        break;
                    }
                }
                if (quiet) {
                    if (lane == 0) cs.ci[ci].nsupp = e1 - e0;
                    __syncwarp();
                    if (cs.nmoves != nmoves0) {
                        mbase = ci + 1;
                        if (mbase >= nch) break;
                        mask = res_chunks_to_visit<STD>(cs, mbase, nch, (float)lam, rn.rmax, a.n, full);
                    }
                    continue;
                }
            }
        }
        const int k0 = cb + lane * SCAN_V;
        const bool in = k0 < ldp;                 // the whole quad is inside the padded row
        T acc[SCAN_V] = {T(0), T(0), T(0), T(0)};
        if (in) slice_dot<T>(a.W, ldp, n4, k0, r, acc);
        T bv[SCAN_V] = {T(0), T(0), T(0), T(0)};
        for (int e = e0; e < e1; ++e) {
            const int t = s.idx[e] - k0;
            if (t >= 0 && t < SCAN_V) {
#pragma unroll
                for (int u = 0; u < SCAN_V; ++u)
                    if (u == t) bv[u] = s.val[e];
            }
        }
        // The slice is exact until the chunk's first move.  After it only the
        // coordinates that can still move are formed again, one at a time: the
        // support's and those at zero that the growth since may have carried to
        // the threshold.  More than RES_OPEN of them (about what a slice costs) form
        // the slice again.
        bool fresh = true, gone = false;
        float grow = 0.f;
        unsigned formed_at = cs.nmoves;
        for (;;) {
            const float reach = (float)lam - (grow * (1.0f + 0x1p-10f) +
                                              rn.rmax * (float)(a.n + 64) * 0x1p-21f +
                                              (float)lam * 0x1p-20f);
            T nbv[SCAN_V];
            unsigned mvmask = 0u;
#pragma unroll
            for (int t = 0; t < SCAN_V; ++t) {
                const int k = k0 + t;
                nbv[t] = bv[t];
                if (k >= cursor && k < p && k != j) {
                    if (fresh) {
                        T nb;
                        if constexpr (STD) {
                            nb = soft<T>(acc[t] + bv[t], lam);                 // ||w_k||^2 = 1
                        } else {
                            const T dk = a.diag[k];
                            nb = soft<T>(acc[t] + dk * bv[t], lam) / dk;       // Soft(c, lambda)/S_kk
                        }
                        nbv[t] = nb;
                        if (nb != bv[t]) mvmask |= 1u << t;
                    } else if (bv[t] != T(0) ||
                               !(fabsf((float)acc[t]) * (1.0f + 0x1p-22f) < reach)) {
                        mvmask |= 1u << t;
                    }
                }
            }
            const unsigned bal = __ballot_sync(FULL_MASK, mvmask != 0u);
            if (bal == 0u) break;
            if (STD && !fresh && __reduce_add_sync(FULL_MASK, __popc(mvmask)) > RES_OPEN) {
                if (in) slice_dot<T>(a.W, ldp, n4, k0, r, acc);
                fresh = true;
                grow = 0.f;
                formed_at = cs.nmoves;
                continue;
            }
            const int f = __ffs(bal) - 1;
            const int tf = __ffs(__shfl_sync(FULL_MASK, mvmask, f)) - 1;
            T nb_sel = nbv[0], b_sel = bv[0];
#pragma unroll
            for (int t = 1; t < SCAN_V; ++t)
                if (t == tf) { nb_sel = nbv[t]; b_sel = bv[t]; }
            T nbs = __shfl_sync(FULL_MASK, nb_sel, f);
            const T bs = __shfl_sync(FULL_MASK, b_sel, f);
            const int ks = cb + f * SCAN_V + tf;
            cursor = ks + 1;
            T v[RES_ROW];
            if (row_in_registers<T, STD>() && a.stage) load_row<T>(a, ks, v);
            if constexpr (STD) {
                if (!fresh) {
                    nbs = soft<T>(coordinate_dot<T>(a, ks, v, stage, r) + bs, lam);
                    if (nbs == bs) {
                        if (cursor >= cb + CHUNK) break;
                        continue;
                    }
                }
            }
            const T delta = nbs - bs;
            int pos = e0;
            while (pos < e1 && s.idx[pos] < ks) ++pos;
            const int n_before = s.n;
            if (!support_set<T>(s, pos, ks, nbs)) {
                overflow = true;
                return maxd;
            }
            e1 += s.n - n_before;
            if (lane == f) {
#pragma unroll
                for (int u = 0; u < SCAN_V; ++u)
                    if (u == tf) bv[u] = nbs;
            }
            maxd = fmax(maxd, fabs(delta));
            ++moves;
            note_residual_move<T, STD>(r, ks, a, v, delta, cs, rn);
            fresh = false;
            gone |= nbs == T(0);
            if constexpr (STD) grow += fabsf((float)delta) * chunk_bound(a, ks, ci);
            if (cursor >= cb + CHUNK) break;
            if constexpr (!STD) {                 // no bounds: the slice again at once
                if (in) slice_dot<T>(a.W, ldp, n4, k0, r, acc);
                fresh = true;
            }
        }
        if constexpr (STD) {
            // the summary: the slice as it was formed, and the growth since.  A
            // coordinate that came to zero here moved its own gradient by more
            // than the growth: it marks the chunk.
            float mx = 0.f;
#pragma unroll
            for (int t = 0; t < SCAN_V; ++t) {
                const int k = k0 + t;
                if (k < p && k != j && bv[t] == T(0)) mx = fmaxf(mx, fabsf((float)acc[t]));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL_MASK, mx, o));
            if (lane == 0) cs.ci[ci] = ResChunk{gone ? INFINITY : mx, grow, formed_at, e1 - e0};
            __syncwarp();
            if (cs.nmoves != nmoves0) {
                mbase = ci + 1;
                if (mbase >= nch) break;
                mask = res_chunks_to_visit<STD>(cs, mbase, nch, (float)lam, rn.rmax, a.n, full);
            }
        } else {
            __syncwarp();
        }
    }
    return maxd;
}

// r_j = w_j - sum_{k in support} w_k b_k recomputed from the data in the data
// precision (lanes over samples), sigma_j^2 = ||r_j||^2 summed in FP64
// (Eq. (14): ||x_j - X b_j||^2 / n on the working scale), and in `dr` the
// distance between the new and the running residual.
template <typename T>
__device__ double residual_reset(int j, const Support<T>& s, T* __restrict__ r,
                                 const ResArgs<T>& a, double& dr) {
    const int lane = threadIdx.x & 31;
    const T* wj = a.Wt + (size_t)j * a.ldn;
    double q = 0.0, d2 = 0.0;
    for (int i = lane; i < a.n; i += 32) {
        T v = wj[i];
#pragma unroll 4
        for (int e = 0; e < s.n; ++e) v = fma(-s.val[e], a.Wt[(size_t)s.idx[e] * a.ldn + i], v);
        const double dv = (double)v;
        q = fma(dv, dv, q);
        const double dd = dv - (double)r[i];
        d2 = fma(dd, dd, d2);
        r[i] = v;
    }
    q = warp_sum(q);
    d2 = warp_sum(d2);
    __syncwarp();
    dr = sqrt(d2);
    return q;
}

// Algorithm 1 for column j in the residual form.
template <typename T, bool STD>
__device__ void solve_column_residual(int j, unsigned char* wsm, const ResArgs<T>& a,
                                      ColCounters& cnt) {
    const int lane = threadIdx.x & 31;
    T* r = reinterpret_cast<T*>(wsm);
    Support<T> s;
    s.idx = reinterpret_cast<int*>(wsm + (size_t)a.ldn * sizeof(T));
    s.val = reinterpret_cast<T*>(s.idx + LAZY_CAP);
    s.n = 0;
    ResScan cs{reinterpret_cast<ResChunk*>(s.val + LAZY_CAP), 0u};
    {
        // b = 0: g_k = w_k' w_j, bounded per chunk by the table
        const int nch = num_chunks(a.ldp);
        for (int c = lane; c < nch; c += 32)
            cs.ci[c] = ResChunk{STD ? chunk_bound(a, j, c) : INFINITY, 0.f, 0u, 0};
    }
    T* stage = reinterpret_cast<T*>(cs.ci + num_chunks(a.ldp));
    // r_j = w_j (b = 0); rows of Wt are zero past n
    const T* wj = a.Wt + (size_t)j * a.ldn;
    double q0 = 0.0;
    for (int i = lane; i < a.ldn; i += 32) {
        const T v = wj[i];
        r[i] = v;
        q0 = fma((double)v, (double)v, q0);
    }
    q0 = warp_sum(q0);
    __syncwarp();
    ResNorm rn;
    rn.rb = (float)sqrt(q0) * (1.0f + 0x1p-20f);
    rn.rmax = rn.rb;

    double sigma = 1.0;                                  // sigma^(0) = 1, b = 0
    const unsigned long long sweeps0 = cnt.sweeps;
    const double floor2 = 1e-12 * q0;                    // S_jj of the working matrix
    int status = COL_OK;
    bool overflow = false;
    int it;
    for (it = 0; it < a.maxit; ++it) {
        const T lam = (T)(sigma * a.lambda0);
        bool inner_ok = false;
        for (int m = 0; m < a.maxit; ++m) {
            const T md = sweep_residual<T, STD>(j, s, r, stage, a, lam, cnt.moves, cs, rn, overflow);
            ++cnt.sweeps;
            if (overflow) break;
            if ((double)md < a.tol) {
                inner_ok = true;
                break;
            }
        }
        if (overflow) {
            status |= COL_NOT_CONVERGED;          // support above the list's capacity
            break;
        }
        if (!inner_ok) status |= COL_NOT_CONVERGED;
        double dr;
        double q = residual_reset<T>(j, s, r, a, dr);
        // the recomputed residual moved r by dr: one move of that size for the
        // skip bound
        for (int c = lane; c < num_chunks(a.ldp); c += 32)
            cs.ci[c].grow += (float)dr * (1.0f + 0x1p-8f);
        ++cs.nmoves;
        __syncwarp();
        rn.rb = (float)sqrt(q) * (1.0f + 0x1p-20f);
        rn.rmax = fmaxf(rn.rmax, rn.rb);
        if (q <= floor2) {
            q = floor2;
            status |= COL_DEGENERATE;
        }
        const double sn = sqrt(q);
        const double ds = fabs(sn - sigma);
        sigma = sn;
        if (ds < a.tol) break;
    }
    if (it == a.maxit) {
        it = a.maxit - 1;
        status |= COL_NOT_CONVERGED;
    }
    T* brow = a.BT + (size_t)j * a.ldp;
    for (int t = lane; t < s.n; t += 32) brow[s.idx[t]] = s.val[t];
    if (lane == 0) {
        a.sigma[j] = sigma;
        a.col_status[j] = status;
    }
    cnt.outer_max = max(cnt.outer_max, it + 1);
    cnt.max_sw = max(cnt.max_sw, (int)(cnt.sweeps - sweeps0));
    cnt.n_nc += (status & COL_NOT_CONVERGED) != 0;
    cnt.n_deg += (status & COL_DEGENERATE) != 0;
    __syncwarp();
}

template <typename T, bool STD>
__global__ void __launch_bounds__(256) cd_residual_kernel(ResArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    unsigned char* wsm = smem_raw + (size_t)warp * (res_warp_smem_bytes<T>(a.ldn, a.ldp) +
                                                    (a.stage ? a.ldn * sizeof(T) : 0));
    FitCtrl* ctrl = a.ctrl;
    if (*reinterpret_cast<volatile int*>(&ctrl->err) != 0) return;
    ColCounters cnt;
    for (;;) {
        int j = 0;
        if (lane == 0) j = atomicAdd(&ctrl->next_col, 1);
        j = __shfl_sync(FULL_MASK, j, 0);
        if (j >= a.p) break;
        solve_column_residual<T, STD>(j, wsm, a, cnt);
    }
    flush_counters(ctrl, cnt);
}

// Per column k (32 columns a 32 x 8 block, see column_means): mu_k (0 without
// centring), s_kk = ||x_k - mu_k||^2 / n
// in FP64, c_k = s_kk^-1/2 when standardising (else 1), the factor
// c_k / sqrt(n) that makes w_k, the working diagonal ||w_k||^2 = c_k^2 s_kk,
// and the starting sigma = 1.  Non-finite data or s_kk <= 0 sets
// DEV_ERR_NONFINITE.  Threads run along k, so every read of X is coalesced.
template <typename T>
__global__ void res_stats_kernel(const T* __restrict__ X, int n, int p, int ldx, int center,
                                 int standardize, double* __restrict__ cs,
                                 double* __restrict__ mu, double* __restrict__ wscale,
                                 T* __restrict__ diag, double* __restrict__ sigma,
                                 int* __restrict__ col_status, FitCtrl* ctrl) {
    __shared__ double part[MEAN_GROUPS][33];
    __shared__ double mean[32];
    const int k = blockIdx.x * 32 + threadIdx.x;
    double m = 0.0;
    if (center) {
        if (k < p) {
#pragma unroll 8
            for (int i = threadIdx.y; i < n; i += MEAN_GROUPS) m += (double)X[(size_t)i * ldx + k];
        }
        m = group_sum(m, part) / (double)n;
        if (threadIdx.y == 0) mean[threadIdx.x] = m;
        __syncthreads();
        m = mean[threadIdx.x];
    }
    double ss = 0.0;
    if (k < p) {
#pragma unroll 8
        for (int i = threadIdx.y; i < n; i += MEAN_GROUPS) {
            const double d = (double)X[(size_t)i * ldx + k] - m;
            ss = fma(d, d, ss);
        }
    }
    ss = group_sum(ss, part);
    if (threadIdx.y != 0 || k >= p) return;
    const double skk = ss / (double)n;
    if (!(skk > 0.0) || !isfinite(skk) || !isfinite(m)) set_error(ctrl, DEV_ERR_NONFINITE);
    const double c = standardize ? 1.0 / sqrt(skk) : 1.0;
    cs[k] = c;
    mu[k] = m;
    wscale[k] = c / sqrt((double)n);
    diag[k] = (T)(c * c * skk);
    sigma[k] = 1.0;
    col_status[k] = COL_OK;
}

// W[i][k] and Wt[k][i] = (x_ik - mu_k) c_k / sqrt(n), formed in FP64 and
// rounded once, over 32 x 32 tiles of (sample, column) that cover the padded
// extents (ldn rows of W, ldn entries of each row of Wt, ldp columns of W),
// with zeros in the padding.  The transpose goes through shared memory so
// that both stores are coalesced.
template <typename T>
__global__ void res_build_kernel(const T* __restrict__ X, int n, int p, int ldx,
                                 const double* __restrict__ mu,
                                 const double* __restrict__ wscale, T* __restrict__ W, int ldp,
                                 T* __restrict__ Wt, int ldn, FitCtrl* ctrl) {
    __shared__ T tile[32][33];
    if (*reinterpret_cast<volatile int*>(&ctrl->err) != 0) return;
    const int i0 = blockIdx.y * 32, k0 = blockIdx.x * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;      // 32 x 8
    const int k = k0 + tx;
    double m = 0.0, sc = 0.0;
    if (k < p) {
        m = mu[k];
        sc = wscale[k];
    }
    for (int rr = ty; rr < 32; rr += 8) {
        const int i = i0 + rr;
        T v = T(0);
        if (i < n && k < p) v = (T)(((double)X[(size_t)i * ldx + k] - m) * sc);
        tile[rr][tx] = v;
        if (i < ldn && k < ldp) W[(size_t)i * ldp + k] = v;
    }
    __syncthreads();
    const int i = i0 + tx;
    for (int rr = ty; rr < 32; rr += 8) {
        const int kk = k0 + rr;
        if (kk < p && i < ldn) Wt[(size_t)kk * ldn + i] = tile[tx][rr];
    }
}

// The bounds of chunk_bound: one block of 128 threads forms 64 columns j against
// the chunks of one byte in FP32, 8 x 8 products a thread, and keeps only the
// row maxima; n 2^-23 covers the rounding of the dots (and of W to FP32).
// Bound by the FP32 pipe: p = 2000, n = 200 0.05 ms.
constexpr int CM_BJ = 64, CM_BK = 16, CM_THREADS = 128;
template <typename T>
__global__ void __launch_bounds__(CM_THREADS) res_cmax_kernel(const T* __restrict__ W, int n, int p,
                                                             int ldp, int cm_chunks,
                                                             unsigned char* __restrict__ cmax0,
                                                             unsigned char* __restrict__ cmax1,
                                                             FitCtrl* ctrl) {
    if (*reinterpret_cast<volatile int*>(&ctrl->err) != 0) return;
    __shared__ __align__(16) float As[CM_BK][CM_BJ], Bs[CM_BK][CHUNK];
    const int g = blockIdx.x, j0 = blockIdx.y * CM_BJ;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;     // 16 x 8
    const int c_end = min((g + 1) * cm_chunks, num_chunks(ldp));
    float m[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) m[u] = 0.f;
    for (int c = g * cm_chunks; c < c_end; ++c) {
        const int k0 = c * CHUNK;
        float acc[8][8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
#pragma unroll
            for (int v = 0; v < 8; ++v) acc[u][v] = 0.f;
        for (int i0 = 0; i0 < n; i0 += CM_BK) {
#pragma unroll
            for (int q = 0; q < CM_BK * CM_BJ / CM_THREADS; ++q) {
                const int e = threadIdx.x + q * CM_THREADS, i = i0 + e / CM_BJ, col = j0 + e % CM_BJ;
                As[e / CM_BJ][e % CM_BJ] = (i < n && col < ldp) ? (float)W[(size_t)i * ldp + col] : 0.f;
            }
#pragma unroll
            for (int q = 0; q < CM_BK; ++q) {
                const int i = i0 + q, col = k0 + threadIdx.x;
                Bs[q][threadIdx.x] = (i < n && col < ldp) ? (float)W[(size_t)i * ldp + col] : 0.f;
            }
            __syncthreads();
#pragma unroll
            for (int kk = 0; kk < CM_BK; ++kk) {
                float a[8], b[8];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    *reinterpret_cast<float4*>(a + 4 * h) =
                        *reinterpret_cast<const float4*>(&As[kk][32 * h + 4 * ty]);
                    *reinterpret_cast<float4*>(b + 4 * h) =
                        *reinterpret_cast<const float4*>(&Bs[kk][64 * h + 4 * tx]);
                }
#pragma unroll
                for (int u = 0; u < 8; ++u)
#pragma unroll
                    for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
            }
            __syncthreads();
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int j = j0 + 32 * (u >> 2) + 4 * ty + (u & 3);
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const int k = k0 + 64 * (v >> 2) + 4 * tx + (v & 3);
                if (k != j) m[u] = fmaxf(m[u], fabsf(acc[u][v]));
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int j = j0 + 32 * (u >> 2) + 4 * ty + (u & 3);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) m[u] = fmaxf(m[u], __shfl_xor_sync(FULL_MASK, m[u], o));
        if (tx == 0 && j < p) {
            const float b = m[u] * (1.0f + 0x1p-20f) + (float)(n + 4) * 0x1p-23f;   // at most 1.003
            (g < 8 ? cmax0 + g : cmax1 + (g - 8))[8 * (size_t)j] =
                (unsigned char)fminf(ceilf(b * 254.0f), 255.0f);
        }
    }
}

template <typename T>
__global__ void res_theta_kernel(const T* __restrict__ BT, int p, int ldp,
                                 const double* __restrict__ sigma, const double* __restrict__ cs,
                                 double* __restrict__ Theta, double* __restrict__ sigma_out,
                                 FitCtrl* ctrl) {
    if (*reinterpret_cast<volatile int*>(&ctrl->err) != 0) return;
    theta_pair<T>(BT, p, ldp, sigma, cs, Theta, sigma_out, ctrl, blockIdx.x);
}

template <typename T, bool STD>
cudaError_t run_residual(const ResLaunch& f, const ResLayout& L, cudaStream_t st) {
    int dev = 0, nsm = 0, smem_optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    unsigned char* ws = f.ws;
    FitCtrl* ctrl = reinterpret_cast<FitCtrl*>(ws + L.ctrl);
    ResArgs<T> a;
    a.W = reinterpret_cast<const T*>(ws + L.W);
    a.Wt = reinterpret_cast<const T*>(ws + L.Wt);
    a.BT = reinterpret_cast<T*>(ws + L.BT);
    a.diag = reinterpret_cast<const T*>(ws + L.diag);
    a.cmax0 = ws + L.mu;
    a.cmax1 = ws + L.wscale;
    a.cm_chunks = (num_chunks(L.ldp) + CM_GROUPS - 1) / CM_GROUPS;
    a.sigma = reinterpret_cast<double*>(ws + L.sigma);
    a.col_status = reinterpret_cast<int*>(ws + L.col_status);
    a.ctrl = ctrl;
    a.n = f.n;
    a.ldn = L.ldn;
    a.p = f.p;
    a.ldp = L.ldp;
    a.maxit = f.maxit;
    a.lambda0 = f.lambda0;
    a.tol = f.tol;
    double* cs = reinterpret_cast<double*>(ws + L.cs);

    size_t per = res_warp_smem_bytes<T>(L.ldn, L.ldp);
    const size_t budget = (size_t)smem_optin - 1024;
    if (per > budget) return cudaErrorInvalidValue;
    a.stage = f.n <= 32 * RES_ROW && per + L.ldn * sizeof(T) <= budget;
    if (a.stage) per += L.ldn * sizeof(T);
    int LW = f.warps_per_block > 0 ? f.warps_per_block : 8;
    LW = std::max(1, std::min({LW, 8, (int)(budget / per)}));
    const size_t smem = per * LW;
    auto kern = cd_residual_kernel<T, STD>;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)smem)) != cudaSuccess)
        return e;
    int per_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * LW, smem)) !=
        cudaSuccess)
        return e;
    per_sm = std::max(per_sm, 1);

    if ((e = cudaMemsetAsync(ctrl, 0, sizeof(FitCtrl), st)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ws + L.BT, 0, (size_t)f.p * L.ldp * sizeof(T), st)) != cudaSuccess)
        return e;
    const T* X = static_cast<const T*>(f.X);
    res_stats_kernel<T><<<(f.p + 31) / 32, dim3(32, MEAN_GROUPS), 0, st>>>(
        X, f.n, f.p, f.ldx, f.center, f.standardize, cs, reinterpret_cast<double*>(ws + L.mu),
        reinterpret_cast<double*>(ws + L.wscale), reinterpret_cast<T*>(ws + L.diag), a.sigma,
        a.col_status, ctrl);
    {
        dim3 grid((L.ldp + 31) / 32, (L.ldn + 31) / 32);
        res_build_kernel<T><<<grid, dim3(32, 8), 0, st>>>(
            X, f.n, f.p, f.ldx, reinterpret_cast<const double*>(ws + L.mu),
            reinterpret_cast<const double*>(ws + L.wscale), reinterpret_cast<T*>(ws + L.W), L.ldp,
            reinterpret_cast<T*>(ws + L.Wt), L.ldn, ctrl);
    }
    if (STD)
        res_cmax_kernel<T><<<dim3((num_chunks(L.ldp) + a.cm_chunks - 1) / a.cm_chunks,
                                  (f.p + CM_BJ - 1) / CM_BJ), CM_THREADS, 0, st>>>(
            a.W, f.n, f.p, L.ldp, a.cm_chunks, ws + L.mu, ws + L.wscale, ctrl);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (f.phase_events) cudaEventRecord(f.phase_events[0], st);
    const int grid = std::min((f.p + LW - 1) / LW, nsm * per_sm);
    kern<<<grid, 32 * LW, smem, st>>>(a);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (f.phase_events) cudaEventRecord(f.phase_events[1], st);
    res_theta_kernel<T><<<theta_pairs<T>(f.p), dim3(32, 8), 0, st>>>(
        a.BT, f.p, L.ldp, a.sigma, cs, f.Theta, f.sigma_out, ctrl);
    if (f.phase_events) cudaEventRecord(f.phase_events[2], st);
    return cudaGetLastError();
}

}  // namespace

bool residual_sizes_ok(int n, int p, int precision) {
    if (n < 1 || n > RES_MAX_N || p < 2) return false;
    const ResLayout L = res_layout(n, p, precision);
    const size_t per = precision == SPMESL_FP64 ? res_warp_smem_bytes<double>(L.ldn, L.ldp)
                                                : res_warp_smem_bytes<float>(L.ldn, L.ldp);
    return per <= 232448 - 1024;
}

cudaError_t launch_fit_residual(const ResLaunch& f, cudaStream_t st) {
    const ResLayout L = res_layout(f.n, f.p, f.precision);
    if (f.precision == SPMESL_FP64)
        return f.standardize ? run_residual<double, true>(f, L, st)
                             : run_residual<double, false>(f, L, st);
    return f.standardize ? run_residual<float, true>(f, L, st)
                         : run_residual<float, false>(f, L, st);
}

}  // namespace spmesl
