// Element operations of the scheme evaluated on the device for tests/test_gpu_device_ops.py: each
// argument row goes through one operation.  Compiled by the test with the flags of the precision's
// kernels (REAL: float or double).
#include "mhd_vjp.cuh"

using R = REAL;
using namespace mhd;

enum Op { GREATER, HLLD_VJP };

__global__ void rows(int op, int nin, int nout, const R* in, R* out, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const R* x = in + (size_t)k * nin;
    R* y = out + (size_t)k * nout;
    const R gamma = R(5.0 / 3.0), gm1i = R(1.5), eps = sizeof(R) == 8 ? R(1e-12) : R(1e-6);
    if (op == GREATER) {
        y[0] = greater_(x[0], x[1]);
    } else if (op == HLLD_VJP) {   // L[7], R[7], bn, cotangents of the flux[5] -> of L, R, bn
        for (int v = 0; v < 15; ++v) y[v] = R(0);
        hlld_vjp(x, x + 7, x[14], gamma, gm1i, eps, x + 15, y, y + 7, y[14]);
    }
}

extern "C" int run_rows(int op, int nin, int nout, const void* in, void* out, int n) {
    rows<<<(n + 127) / 128, 128>>>(op, nin, nout, static_cast<const R*>(in), static_cast<R*>(out), n);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
