// turbulence.cuh -- kernels of the turbulent layer (arXiv 2306.15678, Sec. 3.3,
// Eqs. 9-10): the unnormalised DFTs of row-major arrays (also used by the
// effective lens), with the step spectrum of the random screen formed as they
// read, and the layer's phase
// factor exp(-i thickness eps_t / (2 k0)) on the row-major field.
#pragma once
#include "kernels.cuh"

namespace nlse {

// What a row transform reads: the array itself; the fluence |U|^2 of a field (the
// lens's low-pass); or the spectral amplitude of the turbulent screen, tau xi on
// the bins with p~^2 + q~^2 <= m2max (signed bin numbers; m2max = floor((k_h L / 2
// pi)^2), the same set as comparing the integer p~^2 + q~^2 with the real bound), 0
// elsewhere, rows = k_y.
template <typename T> struct DftLoad {
    const typename vec2<T>::type* a;
    __device__ __forceinline__ typename vec2<T>::type operator()(size_t i, int, int, int) const { return a[i]; }
};
template <typename T> struct DftLoadFluence {
    const typename vec2<T>::type* a;
    __device__ __forceinline__ typename vec2<T>::type operator()(size_t i, int, int, int) const {
        const typename vec2<T>::type u = a[i];
        return mk<typename vec2<T>::type>(u.x * u.x + u.y * u.y, (T)0);
    }
};
template <typename T> struct DftLoadSpectrum {
    const typename vec2<T>::type* a;
    T tau;
    long long m2max;
    __device__ __forceinline__ typename vec2<T>::type operator()(size_t i, int q, int p, int n) const {
        using V = typename vec2<T>::type;
        const long long qq = q < n / 2 ? q : q - n, pp = p < n / 2 ? p : p - n;
        if (pp * pp + qq * qq > m2max) return mk<V>((T)0, (T)0);
        const V v = a[i];
        return mk<V>(tau * v.x, tau * v.y);
    }
};
// What it writes: the array, or the real parts (to `real` and, if given, `real2`),
// with the array too if KEEP
template <typename T> struct DftStore {
    typename vec2<T>::type* a;
    __device__ __forceinline__ void operator()(size_t i, typename vec2<T>::type v) const { a[i] = v; }
};
template <typename T, bool KEEP> struct DftStoreReal {
    typename vec2<T>::type* a;
    T *real, *real2;
    __device__ __forceinline__ void operator()(size_t i, typename vec2<T>::type v) const {
        if (KEEP) a[i] = v;
        if (real) real[i] = v.x;
        if (real2) real2[i] = v.x;
    }
};

// Lines per block of the column transform: adjacent columns are read together,
// so that a warp's loads fill whole 32-byte sectors (4 complex64 or 2
// complex128 columns), within 1024 threads per block; small grids keep the row
// kernels' lines per block.
template <typename T, int N> __host__ __device__ constexpr int dft_cols_per_block() {
    constexpr int TL = threads_per_line<T, N>();
    constexpr int sect = 32 / (2 * (int)sizeof(T));
    constexpr int by_threads = 1024 / TL;
    constexpr int l = sect < by_threads ? sect : by_threads;
    constexpr int rpb = rows_per_block<T, N>();
    return rpb > l ? rpb : l;
}
template <typename T, int N, bool COLS> __host__ __device__ constexpr int dft_lines_per_block() {
    return COLS ? dft_cols_per_block<T, N>() : rows_per_block<T, N>();
}

// Unnormalised DFT (forward, or inverse when INV) of every row of a row-major
// n x n array.  Every line is loaded before the first exchange barrier and stored
// after the last, so the transform may overwrite its input.
template <typename T, int N, bool INV, class LD, class ST>
__global__ void __launch_bounds__(threads_per_line<T, N>() * dft_lines_per_block<T, N, false>(),
                                  min_blocks<threads_per_line<T, N>() * dft_lines_per_block<T, N, false>()>())
k_dft_rows(LD ld, ST st, const typename tab_of<T>::type* __restrict__ tw) {
    using V = typename vec2<T>::type;
    constexpr int E = elems<T, N>(), TL = threads_per_line<T, N>(), LPB = dft_lines_per_block<T, N, false>();
    constexpr int LS = line_stride<T, N, LPB>();
    extern __shared__ __align__(16) unsigned char smraw[];
    const int g = row_of_thread<TL, LPB>(), j = lane_in_row<TL, LPB>();
    const size_t row = (size_t)blockIdx.x * LPB + g;
    V v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = ld(row * N + j + m * TL, (int)row, j + m * TL, N);
    fft_stockham<V, N, E, INV>(v, reinterpret_cast<V*>(smraw) + g * LS, tw, j);
#pragma unroll
    for (int m = 0; m < E; ++m) st(row * N + j + m * TL, v[m]);
}
// The same of every column, in place, and with LOWPASS the forward transform, the
// separable factor fx[p] fy[q] on bin (q, p) (fy carries the 1/n^2 of the inverse
// transforms) and the inverse transform in one sweep (2048^2, cold: 42 us for two
// transforms of 22 and a filter of 12; it spills from 512^2 on, with two transforms
// inlined at 64 registers).  Blocks hold adjacent columns with the column index fastest
// across the threads (coalesced sectors).
template <typename T, int N, bool LOWPASS>
__global__ void __launch_bounds__(threads_per_line<T, N>() * dft_lines_per_block<T, N, true>(),
                                  min_blocks<threads_per_line<T, N>() * dft_lines_per_block<T, N, true>()>())
k_dft_cols(typename vec2<T>::type* data, const typename tab_of<T>::type* __restrict__ tw, const T* __restrict__ fx,
           const T* __restrict__ fy) {
    using V = typename vec2<T>::type;
    constexpr int E = elems<T, N>(), TL = threads_per_line<T, N>(), LPB = dft_lines_per_block<T, N, true>();
    constexpr int LS = line_stride<T, N, LPB>();
    extern __shared__ __align__(16) unsigned char smraw[];
    const int g = (int)(threadIdx.x % LPB), j = (int)(threadIdx.x / LPB);
    const size_t col = (size_t)blockIdx.x * LPB + g;
    V* sm = reinterpret_cast<V*>(smraw) + g * LS;
    V v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = data[col + (size_t)(j + m * TL) * N];
    if constexpr (LOWPASS) {
        fft_stockham<V, N, E, false>(v, sm, tw, j);
        const T f = fx[col];
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = cscale(v[m], f * fy[j + m * TL]);
    }
    fft_stockham<V, N, E, true>(v, sm, tw, j);
#pragma unroll
    for (int m = 0; m < E; ++m) data[col + (size_t)(j + m * TL) * N] = v[m];
}

// The turbulent layer on the row-major field: U <- U exp(-i c Re(eps)),
// c = thickness / (2 k0); the phase and its sine and cosine in the grid
// precision (sincos_ in kernels.cuh).
template <typename T>
__global__ void k_turb_apply(typename vec2<T>::type* field, const typename vec2<T>::type* __restrict__ eps, T c,
                             size_t nn) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nn; i += (size_t)gridDim.x * blockDim.x) {
        T sn, cs;
        sincos_(-c * eps[i].x, &sn, &cs);
        const typename vec2<T>::type u = field[i];
        field[i] = mk<typename vec2<T>::type>(u.x * cs - u.y * sn, u.x * sn + u.y * cs);
    }
}

}  // namespace nlse
