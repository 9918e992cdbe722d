// The node update's reciprocal and square roots on given numbers, beside CUDA's
// correctly rounded ones, for tests/test_gpu_node_math.py.
#include "lbm_kernels.cuh"

enum { RCP, SQRT, SQRT_POS };

template <typename R>
__global__ void evaluate(int fn, int n, const R* a, R* mine, R* cuda) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const R v = a[i];
    mine[i] = fn == RCP ? lbmk::vrcp(v) : fn == SQRT ? lbmk::vsqrt(v) : lbmk::vsqrt_pos(v);
    if constexpr (sizeof(R) == 8) cuda[i] = fn == RCP ? __drcp_rn(v) : __dsqrt_rn(v);
    else cuda[i] = fn == RCP ? __frcp_rn(v) : __fsqrt_rn(v);
}

template <typename R>
static int run(int fn, int n, const R* a, R* mine, R* cuda) {
    R* d = nullptr;
    if (n < 1 || cudaMalloc(&d, 3 * n * sizeof(R)) != cudaSuccess) return 1;
    cudaError_t e = cudaMemcpy(d, a, n * sizeof(R), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        evaluate<R><<<(n + 127) / 128, 128>>>(fn, n, d, d + n, d + 2 * n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(mine, d + n, n * sizeof(R), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(cuda, d + 2 * n, n * sizeof(R), cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? 0 : 1;
}

extern "C" int node_math_f64(int fn, int n, const double* a, double* mine, double* cuda) { return run(fn, n, a, mine, cuda); }
extern "C" int node_math_f32(int fn, int n, const float* a, float* mine, float* cuda) { return run(fn, n, a, mine, cuda); }
