// csrc/fp64_ops.cuh on the device, value by value: host arrays in, host arrays out.
#include "fp64_ops.cuh"

namespace {

__global__ void eval(int n, const double *x, double *rcp, double *drcp, float *cut, const float *f, double *wide) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    rcp[i] = numa::rcp_fp64(x[i]);
    drcp[i] = __drcp_rn(x[i]);
    cut[i] = numa::f64_to_f32_trunc(__double_as_longlong(x[i]));
    wide[i] = numa::f32_to_f64(f[i]);
}

}  // namespace

extern "C" int eval_case(int n, const double *x, const float *f, double *rcp, double *drcp, float *cut, double *wide) {
    double *d = nullptr;   // x, rcp, drcp, wide; cut, f
    float *g = nullptr;
    cudaError_t e = cudaMalloc(&d, sizeof(double) * 4 * n);
    if (e == cudaSuccess) e = cudaMalloc(&g, sizeof(float) * 2 * n);
    if (e == cudaSuccess) e = cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(g + n, f, sizeof(float) * n, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) {
        eval<<<(n + 127) / 128, 128>>>(n, d, d + n, d + 2 * n, g, g + n, d + 3 * n);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(rcp, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(drcp, d + 2 * n, sizeof(double) * n, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(wide, d + 3 * n, sizeof(double) * n, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(cut, g, sizeof(float) * n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    cudaFree(g);
    return (int)e;
}
