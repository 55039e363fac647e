// hot_areas.cuh -- "hot areas" of the beam cross-section (arXiv 2306.15678,
// Sec. 3.3): the closed regions where the fluence w = |U|^2 reaches a cut-off
// w_p, counted as the connected components of the thresholded grid (4 edge
// neighbours, or 8 with the corners; the window is not periodic).
//
// Labelling in four launches over a row-major int32 label array:
//  1. runs:   one block per row labels each pixel with w >= w_p by the index
//             of the first pixel of its horizontal run (block max-scans of
//             run starts over coalesced chunks of the row), every other pixel
//             by -1;
//  2. merge:  the runs of neighbouring rows that touch are joined by a
//             concurrent union-find over the run starts: the larger of two
//             roots is linked under the smaller with atomicMin, and a union
//             that finds its root already linked retries from the new parent;
//  3. roots:  every run start finds its root, compresses its path and counts
//             itself when it is a root;
//  4. spread: every pixel takes the root of its run start.
// Links always point to smaller indices, so every walk ends, and the root of a
// region is its smallest run start, which is its smallest pixel index: the
// labels are unique and equal to a sequential flood fill's, whatever order the
// device joins the runs in.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace nlse {

constexpr int kHotUnionTries = 1 << 20;  // bound on the retries of one union (never reached)
constexpr int kHotStatusGaveUp = 1;      // bit of the per-call status word

// The sweeps take four pixels per thread (16-byte accesses of the labels; n is a
// multiple of 8 and the label array 16-byte aligned): the arrays sit in L2, and with
// one pixel per thread and iteration its latency bounded them (2048^2: runs 19 us,
// merge 18, roots 14, spread 10).

// 1. runs: one block of min(n / 4, 256) threads per row, sweeping the
// row in chunks of 4 blockDim consecutive pixels (coalesced); pixel (y, x) of the
// row-major input is w[(y n + x) stride] (stride 2 reads the real parts of a
// complex array).  A pixel starts a run when it is on and its left neighbour is
// not; its label is the last run start at or before it: a block max-scan of
// the starts within the chunk, carried over from the previous chunks.
template <typename T>
__global__ void __launch_bounds__(256) k_hot_runs(const T* __restrict__ w, int n, int stride, T wp,
                                                  int* __restrict__ label) {
    __shared__ int warp_last[8];
    __shared__ int carry_s;
    const int y = blockIdx.x;
    const T* row = w + (size_t)y * n * stride;
    int* lrow = label + (size_t)y * n;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned mask = blockDim.x >= 32 ? 0xffffffffu : (1u << blockDim.x) - 1u;
    int carry = -1;  // last run start before the chunk
    for (int x0 = 0; x0 < n; x0 += 4 * blockDim.x) {
        const int x = x0 + 4 * threadIdx.x;
        bool on[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) on[q] = row[(size_t)(x + q) * stride] >= wp;
        bool left = x > 0 && row[(size_t)(x - 1) * stride] >= wp;
        int start[4], last = -1;  // last run start of the thread's pixels up to q
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (on[q] && !left) last = x + q;
            start[q] = last;
            left = on[q];
        }
        int incl = last;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(mask, incl, o);
            if (lane >= o) incl = max(incl, v);
        }
        if (lane == 31 || threadIdx.x == blockDim.x - 1) warp_last[warp] = incl;
        int before = __shfl_up_sync(mask, incl, 1);
        if (lane == 0) before = -1;
        __syncthreads();
        before = max(before, carry);
        for (int k = 0; k < warp; ++k) before = max(before, warp_last[k]);
        int4 l;
        l.x = on[0] ? y * n + max(before, start[0]) : -1;
        l.y = on[1] ? y * n + max(before, start[1]) : -1;
        l.z = on[2] ? y * n + max(before, start[2]) : -1;
        l.w = on[3] ? y * n + max(before, start[3]) : -1;
        *reinterpret_cast<int4*>(lrow + x) = l;
        if (threadIdx.x == blockDim.x - 1) carry_s = max(before, last);
        __syncthreads();
        carry = carry_s;
    }
}

// root of pixel i: follow the links (each to a smaller index) to a self-labelled
// run start; reads bypass L1 so that links made by other blocks are seen
__device__ __forceinline__ int hot_find(const int* label, int i) {
    for (;;) {
        const int p = __ldcg(&label[i]);
        if (p == i) return i;
        i = p;
    }
}

__device__ __forceinline__ void hot_union(int* label, int a, int b, int* status) {
    for (int t = 0; t < kHotUnionTries; ++t) {
        a = hot_find(label, a);
        b = hot_find(label, b);
        if (a == b) return;
        if (a > b) {
            const int s = a;
            a = b;
            b = s;
        }
        const int old = atomicMin(&label[b], a);
        if (old == b) return;  // b was still a root: it now hangs under a
        b = old;               // b was linked meanwhile: join a with b's parent instead
    }
    atomicOr(status, kHotStatusGaveUp);
}

__device__ __forceinline__ int hot_at(const int4& v, int q) { return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w; }

// 2. merge: pixel i of rows 0..n-2 joins its run with the runs below it that it
// touches.  With 4 neighbours only the left end of each vertical overlap joins
// (its left neighbours are not both on); with 8, a pixel whose lower neighbour is
// off also joins the runs at its lower corners.  (Only whether a label is
// negative is read here, and no join changes that.)
__global__ void __launch_bounds__(256) k_hot_merge(int* __restrict__ label, int n, int conn, int* __restrict__ status) {
    const int groups = (n - 1) * n / 4;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < groups; g += gridDim.x * blockDim.x) {
        const int i0 = 4 * g, x0 = i0 & (n - 1);
        const int4 up = __ldcg(reinterpret_cast<const int4*>(label + i0));
        if ((up.x & up.y & up.z & up.w) < 0) continue;  // all off
        const int4 dn = __ldcg(reinterpret_cast<const int4*>(label + i0 + n));
        if (conn != 8 && (dn.x & dn.y & dn.z & dn.w) < 0) continue;
        bool up_left = x0 > 0 && __ldcg(&label[i0 - 1]) >= 0, dn_left = x0 > 0 && __ldcg(&label[i0 - 1 + n]) >= 0;
        const bool dn_next = x0 + 4 < n && __ldcg(&label[i0 + 4 + n]) >= 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int i = i0 + q;
            const bool on = hot_at(up, q) >= 0, down = hot_at(dn, q) >= 0;
            const bool right = q < 3 ? hot_at(dn, (q + 1) & 3) >= 0 : dn_next;
            if (on && down) {
                if (!(up_left && dn_left)) hot_union(label, i, i + n, status);
            } else if (on && conn == 8) {
                if (dn_left) hot_union(label, i, i + n - 1, status);
                if (right) hot_union(label, i, i + n + 1, status);
            }
            up_left = on;
            dn_left = down;
        }
    }
}

// 3. roots: the forest is fixed now; every run start finds its root, points
// every start on its path at it, and the roots are counted.  With LENS the slots
// of key and cen of each root are also reset, and it is appended to list, in no
// particular order (list and cen may be null).
template <bool LENS>
__global__ void __launch_bounds__(256) k_hot_roots(int* __restrict__ label, int n, int* __restrict__ count,
                                                   int* __restrict__ list, unsigned long long* __restrict__ key,
                                                   int* __restrict__ cen) {
    const int groups = n * n / 4;
    int local = 0;
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < groups; g += gridDim.x * blockDim.x) {
        const int i0 = 4 * g;
        const int4 l = *reinterpret_cast<const int4*>(label + i0);
        if ((l.x & l.y & l.z & l.w) < 0) continue;  // all off
        bool left = (i0 & (n - 1)) > 0 && label[i0 - 1] >= 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool on = hot_at(l, q) >= 0;
            if (on && !left) {  // a run start
                const int i = i0 + q, r = hot_find(label, i);
                if (r == i) {
                    if constexpr (LENS) {
                        const int at = atomicAdd(count, 1);
                        if (list) list[at] = i;
                        key[i] = 0;
                        if (cen) cen[i] = 0x7fffffff;
                    } else {
                        ++local;
                    }
                }
                for (int s = i; s != r;) {
                    const int p = __ldcg(&label[s]);
                    if (p != r) label[s] = r;
                    s = p;
                }
            }
            left = on;
        }
    }
    if constexpr (!LENS) {
        for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
        if ((threadIdx.x & 31) == 0 && local) atomicAdd(count, local);
    }
}

// 4. spread: every pixel takes its run start's root and hands (root, pixel) to f
struct HotNothing {
    __device__ __forceinline__ void operator()(int, int) const {}
};
template <class F> __global__ void __launch_bounds__(256) k_hot_spread(int* __restrict__ label, int nn, F f) {
    for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < nn / 4; g += gridDim.x * blockDim.x) {
        const int4 l = *reinterpret_cast<const int4*>(label + 4 * g);
        if ((l.x & l.y & l.z & l.w) < 0) continue;  // all off
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int s = hot_at(l, q), i = 4 * g + q;
            if (s < 0) continue;
            const int r = __ldcg(&label[s]);
            if (r != s) label[i] = r;
            f(r, i);
        }
    }
}

}  // namespace nlse
