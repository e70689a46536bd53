// Host entry points around device helpers of libclb, for test_gpu_device_helpers.py.
#include "../paper_1710_10569_gb300/csrc/clb_diag.cuh"

using namespace clb;

namespace {
__global__ void k_doubles(const double* x, double* out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = rcp_halley(x[i]);
    out[n + i] = scale_down<1>(x[i]);
    out[2 * n + i] = scale_down<2>(x[i]);
    out[3 * n + i] = scale_up1(x[i]);
}
__global__ void k_floats(const float* x, double* out, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = widen(x[i]);
}
template <typename T, typename K>
int run(K kernel, const T* x, double* out, int n, int values)
{
    T* dx = nullptr;
    double* dout = nullptr;
    cudaError_t e = cudaMalloc(&dx, n * sizeof(T));
    if (e == cudaSuccess) e = cudaMalloc(&dout, (size_t)values * n * sizeof(double));
    if (e == cudaSuccess) e = cudaMemcpy(dx, x, n * sizeof(T), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        kernel<<<(n + 255) / 256, 256>>>(dx, dout, n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out, dout, (size_t)values * n * sizeof(double), cudaMemcpyDeviceToHost);
    cudaFree(dx);
    cudaFree(dout);
    return (int)e;
}
}  // namespace

extern "C" int helpers_doubles(const double* x, double* out, int n) { return run(k_doubles, x, out, n, 4); }
extern "C" int helpers_floats(const float* x, double* out, int n) { return run(k_floats, x, out, n, 1); }

// A chained launch that the runtime refuses on the host (a grid beyond its limit along y; the kernel's count is
// 0): its error, and the error left behind for the next caller.
extern "C" void helpers_refused_launch(int* refused, int* left)
{
    *refused = (int)launch_chained(k_floats, dim3(1, 70000), dim3(32), 0, nullptr, (const float*)nullptr, (double*)nullptr, 0);
    *left = (int)cudaGetLastError();
}
