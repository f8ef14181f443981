// Gram matrix S = X'X / n: the FP32 path on the CUDA cores and the choice of
// path by precision; the tile itself is in gram_device.cuh.  Only the t(t+1)/2 upper-triangular tiles are
// launched; each writes its mirror too.
#include <cuda_runtime.h>

#include <algorithm>

#include "gram_device.cuh"

namespace spmesl {

namespace {

template <typename T>
__global__ void column_mean_kernel(const T* __restrict__ X, int n, int p, int ldx, T* mu) {
    column_means<T>(X, n, p, ldx, mu, blockIdx.x * 32);
}

template <int BM, int BK, int THREADS, int TM, int TN, bool VEC>
__global__ void __launch_bounds__(THREADS, TM * TN > 64 ? 2 : 4) gram_simt_kernel(const float* __restrict__ X, int n, int p,
                                                           int ldx, const float* __restrict__ mu,
                                                           float* __restrict__ S, int lds,
                                                           float inv_n) {
    int tm, tn;
    upper_tile(blockIdx.x, (p + BM - 1) / BM, tm, tn);
    gram_tile<BM, BK, THREADS, TM, TN, VEC>(X, n, p, ldx, mu, S, lds, inv_n, tm, tn);
}

cudaError_t run_gram_simt(const float* X, int n, int p, int ldx, int center, float* S, int lds,
                          void* ws, cudaStream_t st) {
    float* mu = nullptr;
    if (center) {
        mu = reinterpret_cast<float*>(ws);
        column_mean_kernel<float><<<(p + 31) / 32, dim3(32, MEAN_GROUPS), 0, st>>>(X, n, p, ldx, mu);
    }
    const float inv_n = (float)(1.0 / (double)n);
    const int tw = (p + GRAM_WIDE - 1) / GRAM_WIDE, t = (p + GRAM_BM - 1) / GRAM_BM;
    const bool vec = ((p | ldx) & 3) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0;
    if (tw * (tw + 1) / 2 >= GRAM_WIDE_TILES) {
        auto k = vec ? gram_simt_kernel<GRAM_WIDE, GRAM_WIDE_BK, GRAM_WIDE_THREADS, 8, 16, true>
                     : gram_simt_kernel<GRAM_WIDE, GRAM_WIDE_BK, GRAM_WIDE_THREADS, 8, 16, false>;
        k<<<tw * (tw + 1) / 2, GRAM_WIDE_THREADS, 0, st>>>(X, n, p, ldx, mu, S, lds, inv_n);
    } else {
        auto k = vec ? gram_simt_kernel<GRAM_BM, GRAM_BK, GRAM_THREADS, 8, 4, true>
                     : gram_simt_kernel<GRAM_BM, GRAM_BK, GRAM_THREADS, 8, 4, false>;
        k<<<t * (t + 1) / 2, GRAM_THREADS, 0, st>>>(X, n, p, ldx, mu, S, lds, inv_n);
    }
    return cudaGetLastError();
}

}  // namespace

// Defined in gram_tc.cu (split-BF16 tensor-core path).
size_t gram_tc_ws_bytes(int n, int p);
cudaError_t launch_gram_tc(const float* X, int n, int p, int ldx, int center, float* S, int lds,
                           void* ws, cudaStream_t st);
// Defined in gram_f64.cu (FP64 by error-free digit products on the tensor cores).
size_t gram_f64_ws_bytes(int n, int p);
cudaError_t launch_gram_f64(const double* X, int n, int p, int ldx, int center, double* S, int lds,
                            void* ws, cudaStream_t st);

size_t gram_ws_bytes(int n, int p, int precision) {
    if (precision == SPMESL_MIXED) return gram_tc_ws_bytes(n, p);
    if (precision == SPMESL_FP64) return gram_f64_ws_bytes(n, p);
    return align_up((size_t)p * (size_t)elem_size(precision), 256);
}

cudaError_t launch_gram(const void* X, int n, int p, int ldx, int precision, int center, void* S,
                        int lds, void* ws, cudaStream_t st) {
    if (precision == SPMESL_FP64)
        return launch_gram_f64(static_cast<const double*>(X), n, p, ldx, center,
                               static_cast<double*>(S), lds, ws, st);
    if (precision == SPMESL_FP32)
        return run_gram_simt(static_cast<const float*>(X), n, p, ldx, center,
                             static_cast<float*>(S), lds, ws, st);
    return launch_gram_tc(static_cast<const float*>(X), n, p, ldx, center, static_cast<float*>(S),
                          lds, ws, st);
}

}  // namespace spmesl
