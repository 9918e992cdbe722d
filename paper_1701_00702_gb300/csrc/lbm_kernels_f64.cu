// FP64 storage: instantiation of the fused step, fields, diagnostics and init
// kernels, plus the precision-independent diagnostics finalizer.
#include "lbm_launch.cuh"

namespace lbmk {
LBMK_INSTANTIATE(MODE_F64)
LBMK_INSTANTIATE_CONVERT(MODE_F64)

// Fixed-order sum of the per-block partials: thread t adds sum t mod 4 of the
// blocks t / 4, t / 4 + 128, ..., then a shared-memory tree combines the 128
// threads of each sum.
__global__ void diag_finalize(const double* __restrict__ scratch, int nblocks, double nodes, double* __restrict__ out) {
    __shared__ double red[512];
    const int t = threadIdx.x;
    double a = 0.0;
    for (int i = t; i < 4 * nblocks; i += 512) a += scratch[i];
    red[t] = a;
    __syncthreads();
    for (int w = 256; w >= 4; w >>= 1) {
        if (t < w) red[t] += red[t + w];
        __syncthreads();
    }
    if (t < 4) out[t] = t == 2 ? nodes + red[t] : red[t];
}
}  // namespace lbmk
