// Fixed-point sums of csrc/cgkern.cuh behind C calls on host arrays (tests/test_gpu_fx_sums.py).
#include "cgkern.cuh"

namespace gb {
template <typename T>
__global__ void fold_kernel(const T *a, int n, double *out) {
    __shared__ FoldSmem<2> sm;
    const T x = (int)threadIdx.x < n ? a[threadIdx.x] : T(0);
    const T v[2] = {x, -x};
    const double s = fold_block<2>(v, blockDim.x, sm);
    if ((threadIdx.x & 31) == 0 && threadIdx.x < 64) out[threadIdx.x >> 5] = s;
}
__global__ void parts_kernel(const double *a, int n, double *out) {
    const double s = reduce_parts(a, n);
    if (threadIdx.x == 0) out[0] = s;
}

template <typename T, typename F>
int run(const T *a, int n, double *out, int nout, F &&launch) {
    T *d = nullptr;
    double *o = nullptr;
    if (cudaMalloc(&d, n * sizeof(T)) != cudaSuccess) return 1;
    if (cudaMalloc(&o, nout * sizeof(double)) != cudaSuccess) return 1;
    cudaMemcpy(d, a, n * sizeof(T), cudaMemcpyHostToDevice);
    launch(d, o);
    const cudaError_t e = cudaMemcpy(out, o, nout * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(d);
    cudaFree(o);
    return e == cudaSuccess ? 0 : 1;
}
template <typename T>
int fold(const T *a, int n, int threads, double *out) {
    if (n < 1 || n > threads || threads < 64 || threads > kIterThreads || threads % 32) return 1;
    return run(a, n, out, 2, [&](T *d, double *o) { fold_kernel<T><<<1, threads>>>(d, n, o); });
}
}  // namespace gb

// out[0] the sum over a CTA of `threads` threads, out[1] that of the negated values
extern "C" int fx_fold64(const double *a, int n, int threads, double *out) {
    return gb::fold<double>(a, n, threads, out);
}
extern "C" int fx_fold32(const float *a, int n, int threads, double *out) {
    return gb::fold<float>(a, n, threads, out);
}
// the sum of n CTAs' sums by one warp
extern "C" int fx_parts(const double *a, int n, double *out) {
    if (n < 1 || n > 32 * gb::kPartLoads) return 1;
    return gb::run(a, n, out, 1, [&](double *d, double *o) { gb::parts_kernel<<<1, 32>>>(d, n, o); });
}
