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
//  3. roots:  every run start finds its root and points at it; the roots are
//             counted;
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

// The run sweep takes four neighbouring pixels per thread (16-byte accesses of the
// labels; n is a multiple of 8 and the label array 16-byte aligned).  In the sweeps
// that follow a warp takes a strip of 32 P consecutive pixels, reads what is on with
// one load, leaves an empty strip at once, and works on 32 neighbours at a time: the
// arrays sit in L2, whose latency bounds them.  P = 1 while that is one wave of the
// SMs' threads (n <= 512), as the joins of a fragmented mask are chains of dependent
// loads that a thread should not take one after the other; beyond, 4.  (One pixel per
// thread at every size; four neighbouring pixels per thread; this.  A random mask with 8
// neighbours, whole call: 128^2 83, 156, 70 us; 2048^2 602, 688, 380.  A few spots at
// 2048^2: 95, 74, 74.)
constexpr int kHotStrip = 4;
inline int hot_pixels(int n) { return n <= 512 ? 1 : kHotStrip; }
// blocks of 256 threads of those sweeps
inline int hot_blocks(int n) {
    const int b = (n * n / hot_pixels(n) + 255) / 256;
    return b < 152 * 8 ? b : 152 * 8;
}

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
// run start; reads bypass L1 so that links made by other blocks are seen.  On the way
// every other start is linked to its grandparent (atomicMin: a link only ever moves
// to a smaller ancestor, so one that already points at the root stays).
__device__ __forceinline__ int hot_find(int* label, int i) {
    for (;;) {
        const int p = __ldcg(&label[i]);
        if (p == i) return i;
        const int g = __ldcg(&label[p]);
        if (g == p) return p;
        atomicMin(&label[i], g);
        i = g;
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
        if (old == b) {  // b was still a root: it now hangs under a
            // Rows that join at the same time leave a chain as long as the region is
            // tall, and whoever joins later walks all of it.  With everyone who
            // linked walking and halving at once, what is left is logarithmic (a window
            // that is on everywhere, 1024^2, whole call: 245 us without this, 70 with;
            // 2048^2 157, 97).
            hot_find(label, b);
            return;
        }
        b = old;               // b was linked meanwhile: join a with b's parent instead
    }
    atomicOr(status, kHotStatusGaveUp);
}

// Which pixels of the strip at b are on (label not negative; none from end on), as
// this lane needs it: its pixels 32 r + lane, the ones before and the ones after, as
// bits of one word each.  A strip of four is read with one 16-byte load per lane
// (word q holds pixels 4 lane + q), one of one pixel per lane with a plain one.
template <int P> struct Strip {
    unsigned at = 0, left = 0, right = 0;
    int lane;
    bool any;
    __device__ __forceinline__ Strip(const int* label, int b, int end) : lane(threadIdx.x & 31) {
        static_assert(P == 1 || P == 4, "strip");
        if constexpr (P == 4) {  // (end is a multiple of 128 and b below it)
            const int4 l = __ldcg(reinterpret_cast<const int4*>(label + b) + lane);
            any = __any_sync(0xffffffffu, (l.x & l.y & l.z & l.w) >= 0);
            if (!any) return;
            const unsigned w0 = __ballot_sync(0xffffffffu, l.x >= 0), w1 = __ballot_sync(0xffffffffu, l.y >= 0),
                           w2 = __ballot_sync(0xffffffffu, l.z >= 0), w3 = __ballot_sync(0xffffffffu, l.w >= 0);
            const int q = lane & 3;
            at = q == 0 ? w0 : q == 1 ? w1 : q == 2 ? w2 : w3;
            left = q == 0 ? w3 : q == 1 ? w0 : q == 2 ? w1 : w2;
            right = q == 0 ? w1 : q == 1 ? w2 : q == 2 ? w3 : w0;
        } else {
            at = left = right = __ballot_sync(0xffffffffu, b + lane < end && __ldcg(&label[b + lane]) >= 0);
            any = at != 0;
        }
    }
    // pixel p = 32 r + lane is bit p / P of its word; prev, next: the pixels at either end of the strip
    __device__ __forceinline__ bool on(int r) const { return at >> ((32 * r + lane) / P) & 1u; }
    __device__ __forceinline__ bool before(int r, bool prev) const {
        const int p = 32 * r + lane - 1;
        return p < 0 ? prev : left >> (p / P) & 1u;
    }
    __device__ __forceinline__ bool after(int r, bool next) const {
        const int p = 32 * r + lane + 1;
        return p == 32 * P ? next : right >> (p / P) & 1u;
    }
};
// this thread's first strip and the distance to its next
template <int P> __device__ __forceinline__ int strip_first() {
    return (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 32 * P;
}
template <int P> __device__ __forceinline__ int strip_step() { return (int)(gridDim.x * blockDim.x) * P; }

// 2. merge: pixel i of rows 0..n-2 joins its run with the runs below it that it
// touches.  With 4 neighbours only the left end of each vertical overlap joins
// (its left neighbours are not both on); with 8, a pixel whose lower neighbour is
// off also joins the runs at its lower corners.  (Only whether a label is
// negative is read here, and no join changes that.)
template <int P>
__global__ void __launch_bounds__(256) k_hot_merge(int* __restrict__ label, int n, int conn, int* __restrict__ status) {
    const int nn1 = (n - 1) * n, lane = threadIdx.x & 31;
    for (int b = strip_first<P>(); b < nn1; b += strip_step<P>()) {  // (uniform in the warp)
        const Strip<P> up(label, b, nn1);
        if (!up.any) continue;
        const bool up_prev = b > 0 && __ldcg(&label[b - 1]) >= 0, dn_prev = b > 0 && __ldcg(&label[b - 1 + n]) >= 0;
        const bool dn_next = b + 32 * P < nn1 && __ldcg(&label[b + 32 * P + n]) >= 0;
        const Strip<P> dn(label + n, b, nn1);
        if (!dn.any) {  // corners only, at the ends
            if (conn != 8 || !(dn_prev || dn_next)) continue;
        }
#pragma unroll
        for (int r = 0; r < P; ++r) {
            const int i = b + 32 * r + lane, x = i & (n - 1);
            if (up.on(r)) {
                const bool dn_left = x > 0 && dn.before(r, dn_prev);
                if (dn.on(r)) {
                    if (!(dn_left && up.before(r, up_prev))) hot_union(label, i, i + n, status);
                } else if (conn == 8) {
                    if (dn_left) hot_union(label, i, i + n - 1, status);
                    if (x + 1 < n && dn.after(r, dn_next)) hot_union(label, i, i + n + 1, status);
                }
            }
            __syncwarp();
        }
    }
}

// 3. roots: the regions are fixed now; every run start finds its root and points
// at it, and the roots are counted.  With LENS the slots
// of key and cen of each root are also reset (cen may be null).
template <int P, bool LENS>
__global__ void __launch_bounds__(256) k_hot_roots(int* __restrict__ label, int n, int* __restrict__ count,
                                                   unsigned long long* __restrict__ key, int* __restrict__ cen) {
    const int nn = n * n, lane = threadIdx.x & 31;
    int local = 0;
    for (int b = strip_first<P>(); b < nn; b += strip_step<P>()) {  // (uniform in the warp)
        const Strip<P> row(label, b, nn);
        if (!row.any) continue;
        const bool prev = b > 0 && __ldcg(&label[b - 1]) >= 0;
#pragma unroll
        for (int r = 0; r < P; ++r) {
            const int i = b + 32 * r + lane;
            bool root = false;
            if (row.on(r) && !((i & (n - 1)) > 0 && row.before(r, prev))) {  // a run start
                const int t = hot_find(label, i);
                root = t == i;
                if (!root) label[i] = t;
            }
            __syncwarp();
            local += root;
            if (LENS && root) {
                key[i] = 0;
                if (cen) cen[i] = 0x7fffffff;
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
    if (lane == 0 && local) atomicAdd(count, local);
}

// 4. spread: every pixel takes its run start's root and hands (root, pixel) to f
struct HotNothing {
    __device__ __forceinline__ void operator()(int, int) const {}
};
template <int P, class F>
__global__ void __launch_bounds__(256) k_hot_spread(int* __restrict__ label, int nn, F f) {
    const int lane = threadIdx.x & 31;
    for (int b = strip_first<P>(); b < nn; b += strip_step<P>()) {
        if constexpr (P == 4) {  // nothing on
            const int4 l = *(reinterpret_cast<const int4*>(label + b) + lane);
            if (!__any_sync(0xffffffffu, (l.x & l.y & l.z & l.w) >= 0)) continue;
        }
        int s[P], t[P];
#pragma unroll
        for (int r = 0; r < P; ++r) s[r] = b + 32 * r + lane < nn ? label[b + 32 * r + lane] : -1;
#pragma unroll
        for (int r = 0; r < P; ++r) t[r] = s[r] >= 0 ? __ldcg(&label[s[r]]) : -1;
#pragma unroll
        for (int r = 0; r < P; ++r) {
            if (s[r] < 0) continue;
            const int i = b + 32 * r + lane;
            if (t[r] != s[r]) label[i] = t[r];
            f(t[r], i);
        }
    }
}

// sweeps 2 to 4
template <bool LENS, class F>
inline void hot_sweeps(int* label, int n, int conn, int* count, int* status, unsigned long long* key, int* cen,
                       F f, cudaStream_t s) {
    const int blocks = hot_blocks(n);
    auto run = [&](auto pc) {
        constexpr int P = decltype(pc)::value;
        k_hot_merge<P><<<blocks, 256, 0, s>>>(label, n, conn, status);
        k_hot_roots<P, LENS><<<blocks, 256, 0, s>>>(label, n, count, key, cen);
        k_hot_spread<P><<<blocks, 256, 0, s>>>(label, n * n, f);
    };
    if (hot_pixels(n) == 1) run(std::integral_constant<int, 1>{});
    else run(std::integral_constant<int, kHotStrip>{});
}

}  // namespace nlse
