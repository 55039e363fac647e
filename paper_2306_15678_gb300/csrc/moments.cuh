// moments.cuh -- spatial moments of the fluence (arXiv 2306.15678, Eq. 8):
// M(p, q) = sum over the grid of I^p (x^2 + y^2)^q dx^2 on the cell centres
// x_j = (j - n/2 + 1/2) dx, I = |U|^2, with Eq. 8's Q^m = M(m, m).
#pragma once
#include <cuda_runtime.h>

namespace nlse {

constexpr int kMomMax = 8;

struct MomentSpec {
    int count;
    int p[kMomMax], q[kMomMax];
};

// r[c] = x[c]^e, with no multiplication more than the binary method needs; the
// (uniform) branches on e are taken once for all C values
template <int C> __device__ __forceinline__ void upow(const double (&x)[C], int e, double (&r)[C]) {
    if (e <= 2) {
#pragma unroll
        for (int c = 0; c < C; ++c) r[c] = e == 2 ? x[c] * x[c] : e == 1 ? x[c] : 1.0;
        return;
    }
    double s[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
        s[c] = x[c] * x[c];
        r[c] = e & 1 ? x[c] : 1.0;
    }
    bool one = !(e & 1);  // r is still 1
    for (e >>= 1;;) {
        if (e & 1) {
#pragma unroll
            for (int c = 0; c < C; ++c) r[c] = one ? s[c] : r[c] * s[c];
            one = false;
        }
        if (!(e >>= 1)) return;
#pragma unroll
        for (int c = 0; c < C; ++c) s[c] *= s[c];
    }
}

// Per-block FP64 partial sums of every moment (without the dx^2), written to
// partials[block * kMomMax + k]; the host adds the blocks in a fixed order.  FP64
// instructions bound the kernel (4.2 M points at 2048^2, GB300's 5.3e11 per second),
// so a thread keeps to four columns, whose x^2 it has once, takes y^2 once per row,
// and a power takes no multiplication that it does not need: three moments 233 -> 75
// us.  blockDim = min(n / 4, 256).
template <typename T>
__global__ void __launch_bounds__(256) k_moments(const T* __restrict__ flu, int n, double dx, MomentSpec ms,
                                                 double* __restrict__ partials) {
    __shared__ double red[256];
    double acc[kMomMax], xx[4];
#pragma unroll
    for (int k = 0; k < kMomMax; ++k) acc[k] = 0.0;
    const int x = 4 * (blockIdx.x * blockDim.x + threadIdx.x);
    const double half = 0.5 * dx;  // cell centre j: (2 j - n + 1) dx / 2
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const double xc = (double)(2 * (x + c) - n + 1) * half;
        xx[c] = xc * xc;
    }
    for (int y = blockIdx.y; y < n; y += gridDim.y) {
        const double yc = (double)(2 * y - n + 1) * half, yy = yc * yc;
        const T* row = flu + (size_t)y * n + x;
        double I[4], r2[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            I[c] = (double)row[c];
            r2[c] = xx[c] + yy;
        }
#pragma unroll
        for (int k = 0; k < kMomMax; ++k)
            if (k < ms.count) {
                double a[4], b[4];
                upow(I, ms.p[k], a);
                if (ms.q[k] == 0) {
                    acc[k] += (a[0] + a[1]) + (a[2] + a[3]);
                } else {
                    upow(r2, ms.q[k], b);
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[k] = fma(a[c], b[c], acc[k]);
                }
            }
    }
    const size_t block = blockIdx.y * (size_t)gridDim.x + blockIdx.x;
    for (int k = 0; k < ms.count; ++k) {
        red[threadIdx.x] = acc[k];
        __syncthreads();
        for (int s = blockDim.x / 2; s > 0; s >>= 1) {
            if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
            __syncthreads();
        }
        if (threadIdx.x == 0) partials[block * kMomMax + k] = red[0];
        __syncthreads();
    }
}

}  // namespace nlse
