// Element operations of the scheme evaluated on the device for tests/test_gpu_device_ops.py: each
// argument row goes through one operation.  Compiled by the test with the flags of the precision's
// kernels (REAL: float or double).
#include "mhd_vjp.cuh"

using R = REAL;
using namespace mhd;

enum Op { GREATER, HLLD_VJP, COMPARE, MAX0, EMF2D, EMF2D_VJP, ROOTS, HLL_VJP };

__device__ Corner<R> corner_of(const R* x) { return Corner<R>{x[0], x[1], x[2], x[3], x[4], x[5], x[6]}; }
__device__ void to_row(const Corner<R>& c, R* y) {
    const R v[7] = {c.rho, c.p, c.ua, c.ub, c.Ba, c.Bb, c.Be};
    for (int k = 0; k < 7; ++k) y[k] = v[k];
}

__global__ void rows(int op, int nin, int nout, const R* in, R* out, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const R* x = in + (size_t)k * nin;
    R* y = out + (size_t)k * nout;
    const R gamma = R(5.0 / 3.0), gm1i = R(1.5), eps = sizeof(R) == 8 ? R(1e-12) : R(1e-6);
    if (op == GREATER) {
        y[0] = greater_(x[0], x[1]);
    } else if (op == HLLD_VJP || op == HLL_VJP) {   // L[7], R[7], bn, cotangents of the flux[5] -> of L, R, bn
        for (int v = 0; v < 15; ++v) y[v] = R(0);
        if (op == HLLD_VJP) hlld_vjp(x, x + 7, x[14], gamma, gm1i, eps, x + 15, y, y + 7, y[14]);
        else hll_vjp(x, x + 7, x[14], gamma, gm1i, x + 15, y, y + 7, y[14]);
    } else if (op == COMPARE) {   // a, b
        const R a = x[0], b = x[1];
        y[0] = nonneg_(a);
        y[1] = positive_(a);
        y[2] = nonzero_(a);
        y[3] = greater_(a, b);
        y[4] = same_sign_(a, b);
        y[5] = fmax_(a, b);
        y[6] = fmin_(a, b);
        y[7] = minmod_(a, b);
    } else if (op == MAX0) {   // four values
        y[0] = max0_(x[0], x[1], x[2], x[3]);
        y[1] = min0_(x[0], x[1], x[2], x[3]);
    } else if (op == ROOTS) {
        y[0] = rsqrt_(x[0]);
        y[1] = rcp_(x[0]);
        y[2] = rsqrt_near_(x[0]);
        y[3] = rcp_near_(x[0]);
    } else {   // four corners: rho, p, ua, ub, Ba, Bb, Be each
        Corner<R> c[4];
        for (int v = 0; v < 4; ++v) c[v] = corner_of(x + 7 * v);
        if (op == EMF2D) {
            y[0] = emf2d(c[0], c[1], c[2], c[3], gamma);
        } else {   // and the cotangent of the EMF
            Corner<R> g[4] = {};
            emf2d_vjp(c[0], c[1], c[2], c[3], gamma, x[28], g[0], g[1], g[2], g[3]);
            for (int v = 0; v < 4; ++v) to_row(g[v], y + 7 * v);
        }
    }
}

extern "C" int run_rows(int op, int nin, int nout, const void* in, void* out, int n) {
    rows<<<(n + 127) / 128, 128>>>(op, nin, nout, static_cast<const R*>(in), static_cast<R*>(out), n);
    const cudaError_t e = cudaGetLastError();
    return (int)(e != cudaSuccess ? e : cudaDeviceSynchronize());
}
