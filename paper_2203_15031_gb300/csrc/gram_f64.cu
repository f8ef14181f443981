// FP64 Gram S = X'X / n on the tensor cores (SPMESL_FP64).
//
// The FP64 pipe of this part does two fused multiply-adds a clock and SM, the
// tensor cores several thousand BF16 ones, so the products are formed there
// without error (the splitting of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59, 2012).  Column j
// of X (centred if asked) is scaled by its largest magnitude, |x_ij| < 2^E_j,
// and rounded to the integer v_ij = x_ij 2^(55 - E_j), whose seven balanced
// base-256 digits are exact in BF16.  Digit products are integers of at most
// 2^14, and a level L_l = sum over s + t = l of sum_i d_is d_it, l = 0..7, is
// summed by tcgen05.mma in one FP32 accumulator exactly while it stays below
// 2^24: for up to 256 samples that holds for every input in the levels 0 to 3;
// the levels 4 to 7 (weights 2^-32 and below) can pass 2^24 only when nearly
// all digits are extreme and of one sign, and are then off by units that weigh
// less than 2^-50 of the sum.  After at most 256 samples the levels are
// combined as W = sum_l L_l 256^(7-l), two exact 64-bit integers and one
// FP64 rounding, and S_jk = W 2^(E_j + E_k - 70) / n.
//
// What is left out: the rounding of v, 2^-56 of the column's largest value
// a sample, and the digit products of level 8 and beyond (2^-64 of both largest
// values).  Relative to sqrt(S_jj S_kk) the first is a random sum of about
// 2^-56.8 R / sqrt(n), R = 2^E over the column's root mean square, which is at most
// 2 sqrt(n): below the FP64 sum's own error, whatever the tails.  (Without level
// 7 it was 2^-56.3 R_j R_k / sqrt(n): 4 times the FP64 sum's error for Student t
// with 2 degrees at n = 1000, 30 times for log-normal data.)  Where one sample
// outweighs the rest and an entry does not see it, an FP64 sum is closer still: a column
// with non-finite values, extreme exponents or that many small samples (f64_digit_columns) is
// not scaled, every entry of its row and column is an FP64 sum in sample order
// (direct_entries).
//
// Error of an entry off the diagonal relative to sqrt(S_jj S_kk) against 113-bit sums, a CPU
// restatement, rms, against the FP64 sum in sample order: N(0, 1) n = 30 1.5e-17
// (3.4e-17), n = 250 5.4e-18 (3.7e-17); t with 5 degrees, n = 250 6.8e-18 (3.5e-17);
// with 2, n = 1000 9.9e-18 (4.6e-17); log-normal s = 1, n = 1000 6.0e-17 (3.1e-16).
//
// Measured: p = 100, n = 50 29 us against 72 of FP64 fused multiply-adds at the FP64
// pipe's rate (1.84e9, 0.58 T/s), p = 1500, n = 1000 222 us against 2050, 50 fits of
// p = 500, n = 250 in one launch 0.23 ms with the digits against 3.21.  (Seven levels,
// an instruction per pair of digits: 30, 259 us and 0.26 ms; eight levels so 0.28.)
//
// Kernel: persistent, one CTA of 10 warps per SM over 128 x 64 tiles that hold
// an entry of the upper triangle.  Eight 64-column accumulators fill the
// tensor memory, which sets the tile.  Per K block of 32 samples, warp 0 loads the seven digit planes of the
// tile's rows and columns (two TMA boxes, 84 KB, 64-byte swizzle, two stages);
// one lane of warp 1 issues the 34 digit products of each 16 samples as 12 instructions
// over neighbouring planes (an instruction of one 64-column plane waits for its 6 KB of
// operands longer than for its products); warps 2 to 9
// combine the levels, 32 rows x 32 columns each, hand the accumulators back,
// and write the tile and its mirror while the next tile's products run.
// Waits, failure and tensor-memory release as in gram_tc.cu.  More than F64_SLAB samples
// are a pair of launches (digits, products) for each F64_SLAB of them.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "gram_device.cuh"
#include "gram_f64.cuh"
#include "tc_ptx.cuh"

namespace spmesl {

namespace {

constexpr int F64_THREADS = 320;
constexpr int F64_EPI_WARPS = 8;
constexpr int F64_KB = 32;                            // samples per stage (64-byte rows)
constexpr int F64_STAGES = 2;
constexpr int F64_FLUSH = 256;                        // samples per accumulation
constexpr int F64_RING = 8;
constexpr int F64_A_PLANE = TC_BM * F64_KB * 2;
constexpr int F64_B_PLANE = F64_BN * F64_KB * 2;
constexpr int F64_STAGE_BYTES = F64_SLICES * (F64_A_PLANE + F64_B_PLANE);
constexpr int F64_EPI_COLS = 16;                      // columns staged per store pass
constexpr int F64_EPI_BYTES = 32 * F64_EPI_COLS * 8;  // per epilogue warp
constexpr int F64_TMEM_COLS = 512;
// barriers: full[STAGES], empty[STAGES], acc_full, acc_empty, done
constexpr int F64_NBARS = 2 * F64_STAGES + 3;
constexpr size_t F64_SMEM = (size_t)F64_STAGES * F64_STAGE_BYTES + F64_EPI_WARPS * F64_EPI_BYTES +
                            F64_NBARS * 8 + 64 + 1024;
static_assert(F64_SMEM <= 232448, "shared memory of one block");
static_assert(F64_LEVELS * F64_BN <= F64_TMEM_COLS, "tensor memory");
static_assert(F64_SLICES == 7 && F64_LEVELS == 8, "the products are listed for these");
static_assert(F64_FLUSH % F64_KB == 0 && TC_NPAD % F64_KB == 0, "K blocks");
// instruction descriptor: BF16 x BF16 -> FP32, both K-major, M = 128, N = m digit
// planes of F64_BN columns
__host__ __device__ constexpr unsigned f64_idesc(int m) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)((m * F64_BN) >> 3) << 17) |
           ((unsigned)(TC_BM >> 4) << 24);
}

// Shared-memory descriptor of a K-major operand plane with 64-byte rows and
// 64-byte swizzle (8-row groups 512 bytes apart; planes start on 512 bytes).
__device__ __forceinline__ unsigned long long plane_desc(unsigned addr) {
    unsigned long long d = 0;
    d |= (unsigned long long)((addr & 0x3FFFFu) >> 4);
    d |= (unsigned long long)1 << 16;
    d |= (unsigned long long)((8 * F64_KB * 2) >> 4) << 32;
    d |= (unsigned long long)1 << 46;
    d |= 4ull << 61;
    return d;
}

__device__ __forceinline__ void mma_digits(unsigned tmem_d, unsigned long long a,
                                           unsigned long long b, unsigned idesc,
                                           unsigned accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap* map, int x, int y,
                                            int z, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

struct F64One {
    F64Fit f;
    int n_tiles, s0;
    static constexpr bool kTableMaps = false;
    __device__ int tiles() const { return n_tiles; }
    __device__ int fits() const { return 1; }
    __device__ int fit_index(int) const { return 0; }
    __device__ const F64Fit& fit_at(int) const { return f; }
    __device__ const int* marks() const { return f.marks; }
    __device__ int n_marks() const { return (f.p + 31) / 32; }
    __device__ int first() const { return s0; }
};

struct F64Many {
    F64Batch b;
    static constexpr bool kTableMaps = true;
    __device__ int tiles() const { return b.n_tiles; }
    __device__ int fits() const { return b.n_fits; }
    __device__ int fit_index(int tile) const { return __ldg(b.tile_fit + tile); }
    __device__ const F64Fit& fit_at(int fi) const { return b.fits[fi]; }
    __device__ const int* marks() const { return b.marks; }
    __device__ int n_marks() const { return b.n_marks; }
    __device__ int first() const { return b.s0; }
};

// K blocks of a fit in the slab that starts at sample s0 (0 or less: it has none), and
// whether it is the fit's last.
__device__ __forceinline__ int slab_blocks(const F64Fit& f, int s0) {
    return min(tc_pad_n(f.n) - s0, F64_SLAB) / F64_KB;
}
__device__ __forceinline__ bool last_slab(const F64Fit& f, int s0) { return f.n - s0 <= F64_SLAB; }

// The entries of rows r0 .. r0 + 31 and columns c0 .. c0 + 63 whose row or column is
// not scaled (F64_EXPO_DIRECT): FP64 sums in sample order.  Bound by the FP64 pipe
// (16 cycles of the SM an instruction of a warp), so a warp's instruction is a group of 32
// entries that are wanted: half a row that is not scaled, or a column that is not scaled
// over the 32 rows; when these come to more than the block's 64 half rows, the half rows.
// Blocks of 32 x 64, in turn over the grid, keep every SM at work: p = 500, n = 250 48 us
// without such columns, 82 with one, 197 with all of them (567 and 624 when each CTA
// formed them for its own 128 x 64 tiles); p = 1500, n = 1000 221, 345 and 2573
// (the products alone take 1.94 ms of the FP64 pipe).
constexpr int F64_DIRECT_BK = 64;
constexpr int F64_DIRECT_WARPS = 8;                   // that form them: 64 groups come out even
constexpr int F64_DIRECT_GROUPS = 64 / F64_DIRECT_WARPS;
static_assert(F64_DIRECT_BK * (32 + F64_BN) * 8 <= F64_STAGES * F64_STAGE_BYTES, "stage buffers");
__device__ __noinline__ void direct_block(const F64Fit& f, int r0, int c0, double* __restrict__ sm) {
    double (*As)[32] = reinterpret_cast<double (*)[32]>(sm);
    double (*Bs)[F64_BN] = reinterpret_cast<double (*)[F64_BN]>(sm + F64_DIRECT_BK * 32);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, p = f.p;
    auto unscaled = [&](int c) { return c < p && f.expo[c] == F64_EXPO_DIRECT; };
    const unsigned rows = __ballot_sync(FULL_MASK, unscaled(r0 + lane));
    const unsigned lo = __ballot_sync(FULL_MASK, unscaled(c0 + lane));
    const unsigned hi = __ballot_sync(FULL_MASK, unscaled(c0 + 32 + lane));
    const int nr = 2 * __popc(rows), nlo = __popc(lo), nc = nlo + __popc(hi);
    const bool half_rows = nr + nc > 64;
    const int groups = half_rows ? 64 : nr + nc;
    int ia[F64_DIRECT_GROUPS], ib[F64_DIRECT_GROUPS], cnt = 0;
    unsigned valid = 0u;
    double acc[F64_DIRECT_GROUPS];
#pragma unroll
    for (int q = 0; q < F64_DIRECT_GROUPS; ++q) {
        const int g = warp + q * F64_DIRECT_WARPS;
        acc[q] = 0.0;
        ia[q] = ib[q] = 0;
        if (warp < F64_DIRECT_WARPS && g < groups) {
            const bool column = !half_rows && g >= nr;
            int r = lane, c = 32 * (g & 1) + lane;
            if (half_rows) r = g >> 1;
            else if (!column) r = (int)__fns(rows, 0, (g >> 1) + 1);
            else if (g - nr < nlo) c = (int)__fns(lo, 0, g - nr + 1);
            else c = 32 + (int)__fns(hi, 0, g - nr - nlo + 1);
            const bool dr = (rows >> r) & 1u, dc = ((c < 32 ? lo : hi) >> (c & 31)) & 1u;
            if (r0 + r < p && c0 + c < p && c0 + c >= r0 + r && (dr || dc) && !(column && dr))
                valid |= 1u << q;
            ia[q] = r;
            ib[q] = c;
            cnt = q + 1;
        }
    }
    for (int i0 = 0; i0 < f.n; i0 += F64_DIRECT_BK) {
        const int nk = min(F64_DIRECT_BK, f.n - i0);
        __syncthreads();                      // the last samples' readers are done
#pragma unroll 4
        for (int e = tid; e < nk * (32 + F64_BN); e += F64_THREADS) {
            const int kk = e / (32 + F64_BN), c = e % (32 + F64_BN);
            const int col = c < 32 ? r0 + c : c0 + c - 32;
            const double x = col < p ? f.X[(size_t)(i0 + kk) * f.ldx + col] - (f.mu ? f.mu[col] : 0.0)
                                     : 0.0;
            if (c < 32) As[kk][c] = x;
            else Bs[kk][c - 32] = x;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < F64_DIRECT_GROUPS; ++q) {
            if (q >= cnt) break;
#pragma unroll 4
            for (int kk = 0; kk < nk; ++kk) acc[q] = fma(As[kk][ia[q]], Bs[kk][ib[q]], acc[q]);
        }
    }
#pragma unroll
    for (int q = 0; q < F64_DIRECT_GROUPS; ++q)
        if ((valid >> q) & 1u) {
            const size_t row = r0 + ia[q], col = c0 + ib[q];
            const double s = acc[q] * f.inv_n;
            f.S[row * f.lds + col] = s;
            f.S[col * f.lds + row] = s;
        }
    __syncthreads();
}

// Blocks of direct_block that hold an entry of the upper triangle: the two halves
// of each 64 x 64 tile.
__host__ __device__ inline int direct_blocks(int p) {
    const int t = (p + 63) / 64;
    return t * (t + 1);
}

// All such entries of all fits, their blocks in turn over the grid (each entry is
// written here only): after the CTA's last tile, when no role waits, since they take n
// times the epilogue's work.  32 blocks are looked at at once, by every warp alike.
template <class Src>
__device__ __forceinline__ void direct_entries(const Src& src, double* sm) {
    const int lane = threadIdx.x & 31, G = gridDim.x;
    int first = blockIdx.x;                   // of the fit's blocks, modulo G
    for (int fi = 0; fi < src.fits(); ++fi) {
        const F64Fit& f = src.fit_at(fi);
        if (f.p == 0 || f.n <= src.first() || !last_slab(f, src.first())) continue;
        const int nm = (f.p + 31) / 32, t = (f.p + 63) / 64, nb = direct_blocks(f.p);
        bool any = false;
        for (int i = lane; i < nm; i += 32) any |= f.marks[i] != 0;
        if (__any_sync(FULL_MASK, any)) {
            for (int s0 = first; s0 < nb; s0 += 32 * G) {
                const long long s = s0 + (long long)lane * G;
                int tm = 0, tn = 0;
                bool hit = false;
                if (s < nb) {
                    upper_tile((int)(s >> 1), t, tm, tn);
                    const int rb = 2 * tm + (int)(s & 1);
                    hit = rb < nm && (f.marks[rb] || f.marks[2 * tn] ||
                                      (2 * tn + 1 < nm && f.marks[2 * tn + 1]));
                }
                unsigned left = __ballot_sync(FULL_MASK, hit);
                for (; left; left &= left - 1u) {
                    const int l = __ffs(left) - 1;
                    const int rm = __shfl_sync(FULL_MASK, tm, l), rn = __shfl_sync(FULL_MASK, tn, l);
                    direct_block(f, 64 * rm + 32 * ((s0 + l * G) & 1), 64 * rn, sm);
                }
            }
        }
        first = (first + G - nb % G) % G;
    }
}

// W = L_0 256^7 + .. + L_7 from the eight integer-valued level sums: the
// upper and the lower four levels as 64-bit integers (below 2^50), made
// FP64 by the 1.5 2^52 offset, and one rounding.
__device__ __forceinline__ double combine_levels(const unsigned (&L)[F64_LEVELS][8], int c) {
    auto I = [&](int l) { return (long long)__float2int_rn(__uint_as_float(L[l][c])); };
    const long long hi = ((I(0) * 256 + I(1)) * 256 + I(2)) * 256 + I(3);
    const long long lo = ((I(4) * 256 + I(5)) * 256 + I(6)) * 256 + I(7);
    const double off = 6755399441055744.0;
    const double h = __longlong_as_double(0x4338000000000000ll + hi) - off;
    const double l = __longlong_as_double(0x4338000000000000ll + lo) - off;
    return fma(h, 4294967296.0, l);
}

template <class Src>
__global__ void __launch_bounds__(F64_THREADS, 1) gram_f64_kernel(const __grid_constant__ Src src) {
    extern __shared__ unsigned char smem_dyn[];
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~(uintptr_t)1023);
    unsigned char* stages = smem;
    double* epi = reinterpret_cast<double*>(smem + (size_t)F64_STAGES * F64_STAGE_BYTES);
    unsigned long long* bars = reinterpret_cast<unsigned long long*>(
        smem + (size_t)F64_STAGES * F64_STAGE_BYTES + F64_EPI_WARPS * F64_EPI_BYTES);
    unsigned long long* full = bars;
    unsigned long long* empty = bars + F64_STAGES;
    unsigned long long* acc_full = bars + 2 * F64_STAGES;
    unsigned long long* acc_empty = acc_full + 1;
    unsigned long long* done = acc_full + 2;
    volatile unsigned* tmem_slot = reinterpret_cast<volatile unsigned*>(bars + F64_NBARS);
    volatile int* fail = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* issued_slot = fail + 1;
    volatile int* consumed_slot = fail + 2;
    volatile int* direct_slot = fail + 3;     // some column of the CTA's tiles is not scaled
    volatile int* kt_ring = fail + 4;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_tiles = src.tiles(), s0 = src.first();

    if (threadIdx.x == 0) {
        for (int s = 0; s < F64_STAGES; ++s) {
            mbar_init(smem_u32(&full[s]), 1);
            mbar_init(smem_u32(&empty[s]), 1);
        }
        mbar_init(smem_u32(acc_full), 1);
        mbar_init(smem_u32(acc_empty), F64_EPI_WARPS);
        mbar_init(smem_u32(done), 1);
        *fail = 0;
        *issued_slot = 0;
        *consumed_slot = 0;
        *direct_slot = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(const_cast<unsigned*>(tmem_slot))),
                     "r"(F64_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const unsigned tmem = *tmem_slot;

    if (warp == 0) {
        if (lane == 0) {
            // producer
            int kb = 0, li = 0;
            const F64Fit* last = nullptr;
            for (int tile = blockIdx.x; tile < n_tiles && !*fail; tile += gridDim.x) {
                const F64Fit& f = src.fit_at(src.fit_index(tile));
                const int KT = slab_blocks(f, s0);
                if (KT <= 0) continue;              // a shorter fit of the batch
                int tm, tn;
                f.g.coords(tile - f.tile_start, tm, tn);
                kt_ring[li % F64_RING] = KT;        // published by the first expect_tx below
                if (Src::kTableMaps && &f != last) {
                    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                                     reinterpret_cast<unsigned long long>(&f.ma))
                                 : "memory");
                    asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(
                                     reinterpret_cast<unsigned long long>(&f.mb))
                                 : "memory");
                    last = &f;
                }
                for (int kt = 0; kt < KT; ++kt, ++kb) {
                    const int s = kb % F64_STAGES;
                    if (kb >= F64_STAGES &&
                        !mbar_wait(smem_u32(&empty[s]), ((kb / F64_STAGES) - 1) & 1, fail)) {
                        *fail = 1;
                        break;
                    }
                    const unsigned fb = smem_u32(&full[s]);
                    unsigned char* st = stages + (size_t)s * F64_STAGE_BYTES;
                    mbar_expect_tx(fb, F64_STAGE_BYTES);
                    tma_load_3d(smem_u32(st), &f.ma, kt * F64_KB, tm * TC_BM, 0, fb);
                    tma_load_3d(smem_u32(st + F64_SLICES * F64_A_PLANE), &f.mb, kt * F64_KB,
                                tn * F64_BN, 0, fb);
                    *issued_slot = kb + 1;
                }
                ++li;
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // MMA issuer
            int kb = 0, li = 0, flush = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
                if (s0 != 0 && slab_blocks(src.fit_at(src.fit_index(tile)), s0) <= 0) continue;
                int KT = 1;                          // read once the first K block has landed
                for (int kt = 0; kt < KT; ++kt, ++kb) {
                    const bool first = kt % (F64_FLUSH / F64_KB) == 0;
                    if (first) {
                        if (flush >= 1 && !mbar_wait(smem_u32(acc_empty), (flush - 1) & 1, fail)) {
                            ok = false;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    }
                    const int s = kb % F64_STAGES;
                    if (!mbar_wait(smem_u32(&full[s]), (kb / F64_STAGES) & 1, fail)) {
                        ok = false;
                        break;
                    }
                    if (kt == 0) KT = kt_ring[li % F64_RING];
                    *consumed_slot = kb + 1;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const unsigned base = smem_u32(stages + (size_t)s * F64_STAGE_BYTES);
                    const unsigned long long a0 = plane_desc(base),
                                             b0 = plane_desc(base + F64_SLICES * F64_A_PLANE);
#pragma unroll
                    for (int kk = 0; kk < F64_KB / 16; ++kk) {
                        // 16 bf16 = 32 bytes along K inside the swizzled rows
                        const unsigned long long off = (unsigned long long)((32 * kk) >> 4);
                        // plane t of the rows by planes u .. u + m - 1 of the columns, which follow
                        // one another in shared memory as the levels t + u .. do in tensor memory
                        auto products = [&](int t, int u, int m, bool add) {
                            mma_digits(tmem + (t + u) * F64_BN,
                                       a0 + off + (unsigned long long)((t * F64_A_PLANE) >> 4),
                                       b0 + off + (unsigned long long)((u * F64_B_PLANE) >> 4),
                                       f64_idesc(m), add ? 1u : 0u);
                        };
                        const bool add = !first || kk;
                        products(0, 0, 4, add);
                        products(0, 4, 3, add);
                        products(1, 0, 4, true);
                        products(1, 4, 2, true);
                        products(1, 6, 1, add);            // level 7's first
                        products(2, 0, 4, true);
                        products(2, 4, 2, true);
                        products(3, 0, 3, true);
                        products(3, 3, 2, true);
                        products(4, 0, 4, true);
                        products(5, 0, 3, true);
                        products(6, 0, 2, true);
                    }
                    mma_commit(smem_u32(&empty[s]));
                    if ((kt + 1) % (F64_FLUSH / F64_KB) == 0 || kt + 1 == KT) {
                        mma_commit(smem_u32(acc_full));
                        ++flush;
                    }
                }
                ++li;
            }
            if (!ok) *fail = 1;
            mma_commit(smem_u32(done));
            mbar_wait(smem_u32(done), 0, nullptr);
        }
    } else {
        // epilogue: warp w reads accumulator lanes 32 (w % 4) .. +31, warps 2-5
        // the first half of the columns and warps 6-9 the second
        const int ew = warp - 2;
        const int q = warp & 3, half = ew >> 2;
        double* buf = epi + ew * (F64_EPI_BYTES / 8);     // 32 rows x 16 columns, XOR-swizzled
        for (int i = 32 * ew + lane; i < src.n_marks(); i += 32 * F64_EPI_WARPS)
            if (src.marks()[i]) *direct_slot = 1;
        bool ok = true;
        int flush = 0;
        for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
            const F64Fit& f = src.fit_at(src.fit_index(tile));
            const int KT = slab_blocks(f, s0);
            if (KT <= 0) continue;
            int tm, tn;
            f.g.coords(tile - f.tile_start, tm, tn);
            const int m0 = tm * TC_BM + 32 * q, c0 = tn * F64_BN + 32 * half;
            const int p = f.p, lds = f.lds;
            // warp-uniform: this warp's 32 x 32 block holds an entry to write
            const bool any = m0 < p && c0 < p && c0 + 31 >= m0;
            double acc[32];
            double* __restrict__ S = f.S;
            const int row = m0 + lane;
            if (s0 != 0 && any) {                         // the slabs before this one
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int col = c0 + i;
                    acc[i] = (col < p && col >= row) ? S[(size_t)col * lds + row] : 0.0;
                }
            }
            const int nf = (KT * F64_KB + F64_FLUSH - 1) / F64_FLUSH;
            for (int fl = 0; fl < nf; ++fl, ++flush) {
                if (ok) {
                    int got = 0;
                    if (lane == 0) got = mbar_wait(smem_u32(acc_full), flush & 1, fail) ? 1 : 0;
                    ok = __shfl_sync(FULL_MASK, got, 0) != 0;
                    if (!ok && lane == 0) *fail = 1;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                if (any && ok) {
#pragma unroll
                    for (int c = 0; c < 32; c += 8) {
                        unsigned L[F64_LEVELS][8];
#pragma unroll
                        for (int l = 0; l < F64_LEVELS; ++l)
                            tmem_ld8(tmem + ((unsigned)(32 * q) << 16) +
                                         (unsigned)(l * F64_BN + 32 * half + c),
                                     L[l]);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const double w = combine_levels(L, i);
                            acc[c + i] = (fl == 0 && s0 == 0) ? w : acc[c + i] + w;
                        }
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) mbar_arrive(smem_u32(acc_empty));
            }
            if (!any) continue;
            if (!last_slab(f, s0)) {
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int col = c0 + i;
                    if (col < p && col >= row)
                        S[(size_t)col * lds + row] = ok ? acc[i] : __longlong_as_double(0x7ff8000000000000ll);
                }
                continue;
            }
            const int Ej = row < p ? f.expo[row] : 0;
            // inv_n 2^(E_j - 70); E_k is added to its exponent per column
            const double sj = Ej == F64_EXPO_DIRECT ? f.inv_n : scalbn(f.inv_n, Ej - 70);
            const int my_E = c0 + lane < p ? f.expo[c0 + lane] : 0;
            // rows and columns of the block that direct_entries forms
            const unsigned dr = __ballot_sync(FULL_MASK, Ej == F64_EXPO_DIRECT);
            const unsigned dc = __ballot_sync(FULL_MASK, my_E == F64_EXPO_DIRECT);
            const unsigned skip = Ej == F64_EXPO_DIRECT ? FULL_MASK : dc;
#pragma unroll
            for (int i = 0; i < 32; ++i) {
                const int Ek = __shfl_sync(FULL_MASK, my_E, i);
                if (!ok) {
                    acc[i] = __longlong_as_double(0x7ff8000000000000ll);
                } else {
                    acc[i] *= __longlong_as_double(__double_as_longlong(sj) + ((long long)Ek << 52));
                }
            }
            // the mirror S_kj, lanes along row k
            if (row < p) {
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int col = c0 + i;
                    if (col < p && col > row && !((skip >> i) & 1u)) S[(size_t)col * lds + row] = acc[i];
                }
            }
            // S_jk, two rows of 128 bytes per store, through shared memory
#pragma unroll
            for (int h = 0; h < 32; h += F64_EPI_COLS) {
                __syncwarp();
#pragma unroll
                for (int i = 0; i < F64_EPI_COLS; ++i)
                    buf[lane * F64_EPI_COLS + (i ^ (lane & 15))] = acc[h + i];
                __syncwarp();
                const int col = c0 + h + (lane & 15);
                for (int jj = 0; jj < 32; jj += 2) {
                    const int j = jj + (lane >> 4), r = m0 + j;
                    if (r < p && col < p && col >= r && !((dr >> j) & 1u) &&
                        !((dc >> (h + (lane & 15))) & 1u))
                        S[(size_t)r * lds + col] = buf[j * F64_EPI_COLS + ((lane & 15) ^ (j & 15))];
                }
            }
        }
    }
    __syncthreads();
    if (*fail && threadIdx.x == 0) {
        // let copies still in flight land before the CTA exits (bounded)
        const int issued = *issued_slot, consumed = *consumed_slot;
        for (int kb = consumed; kb < issued; ++kb)
            mbar_wait(smem_u32(&full[kb % F64_STAGES]), (kb / F64_STAGES) & 1, nullptr);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (*direct_slot) direct_entries(src, reinterpret_cast<double*>(stages));   // (idle by now)
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(F64_TMEM_COLS));
    }
}

__global__ void __launch_bounds__(256) f64_digits_kernel(const double* __restrict__ X, int n, int p,
                                                        int ldx, const double* __restrict__ mu,
                                                        int* __restrict__ expo, int* __restrict__ marks,
                                                        __nv_bfloat16* __restrict__ D, int s0) {
    f64_digit_columns(X, n, p, ldx, mu, expo, marks + blockIdx.x, f64_counts(expo, p), D,
                      blockIdx.x * 32, s0);
}

__global__ void f64_mean_kernel(const double* __restrict__ X, int n, int p, int ldx, double* mu) {
    column_means<double>(X, n, p, ldx, mu, blockIdx.x * 32);
}

template <class Src>
cudaError_t launch_tiles(const Src& src, int n_tiles, int n_blocks, cudaStream_t st) {
    auto kern = gram_f64_kernel<Src>;
    cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F64_SMEM);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return e;
    if (n_tiles <= 0) return cudaSuccess;
    // (a CTA without a tile costs little, and the blocks of direct_entries are more than the tiles)
    const int grid = n_tiles > n_blocks ? n_tiles : n_blocks;
    kern<<<grid < sms ? grid : sms, F64_THREADS, F64_SMEM, st>>>(src);
    return cudaGetLastError();
}

}  // namespace

size_t gram_f64_ws_bytes(int n, int p) {
    return align_up((size_t)p * 8, 256) + f64_expo_bytes(p) + f64_digit_bytes(n, p);
}

bool f64_encode_fit(F64Fit& f, const double* X, int n, int p, int ldx, const double* mu,
                    const int* expo, const int* marks, const void* D, double* S, int lds,
                    int tile_start) {
    f = F64Fit{};
    const unsigned long long ldd = f64_plane_n(n);
    const unsigned long long dims[3] = {ldd, (unsigned long long)p, (unsigned long long)F64_SLICES};
    const unsigned long long strides[2] = {ldd * 2, ldd * 2 * p};
    const unsigned box_a[3] = {F64_KB, TC_BM, F64_SLICES}, box_b[3] = {F64_KB, F64_BN, F64_SLICES};
    if (!tc_encode_bf16_3d(f.ma, D, dims, strides, box_a) ||
        !tc_encode_bf16_3d(f.mb, D, dims, strides, box_b))
        return false;
    f.X = X;
    f.mu = mu;
    f.expo = expo;
    f.marks = marks;
    f.S = S;
    f.n = n;
    f.p = p;
    f.ldx = ldx;
    f.lds = lds;
    f.tile_start = tile_start;
    f.inv_n = 1.0 / (double)n;
    f.g = tc_tile_grid(p, F64_BN);
    return true;
}

cudaError_t launch_gram_f64(const double* X, int n, int p, int ldx, int center, double* S, int lds,
                            void* ws, cudaStream_t st) {
    unsigned char* base = static_cast<unsigned char*>(ws);
    double* mu = center ? reinterpret_cast<double*>(base) : nullptr;
    int* expo = reinterpret_cast<int*>(base + align_up((size_t)p * 8, 256));
    __nv_bfloat16* D = reinterpret_cast<__nv_bfloat16*>(base + align_up((size_t)p * 8, 256) +
                                                        f64_expo_bytes(p));
    int* marks = expo + p;
    F64One one;
    if (!f64_encode_fit(one.f, X, n, p, ldx, mu, expo, marks, D, S, lds, 0)) return cudaErrorInvalidValue;
    one.n_tiles = one.f.g.count();
    if (center) f64_mean_kernel<<<(p + 31) / 32, dim3(32, MEAN_GROUPS), 0, st>>>(X, n, p, ldx, mu);
    for (long long s0 = 0; s0 < n; s0 += F64_SLAB) {
        one.s0 = (int)s0;
        f64_digits_kernel<<<(p + 31) / 32, dim3(32, 8), 0, st>>>(X, n, p, ldx, mu, expo, marks, D, one.s0);
        const cudaError_t e = launch_tiles(one, one.n_tiles, direct_blocks(p), st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int f64_direct_blocks(int p) { return direct_blocks(p); }

cudaError_t launch_gram_f64_batch(const F64Batch& b, cudaStream_t st) {
    return launch_tiles(F64Many{b}, b.n_tiles, b.n_blocks, st);
}

}  // namespace spmesl
