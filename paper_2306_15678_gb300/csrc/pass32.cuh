// pass32.cuh -- the FP32 (complex64) march on the pair engine (pair.cuh):
// the two HBM sweeps of a split-step z step (arXiv 2306.15678, Eq. 2 with the
// terms of Eq. 1 and Eq. 3), the load prologue and the readout.
//
// State between steps: S = F_x U in the unit layout of pair.cuh, unit
// (p n + x) = (re, im) of rows 2p and 2p+1 at column x.  One step is
//   column pass: S <- B_y( P_x(kx) P_y(ky) rot / n^2 * F_y S )   (diffraction)
//   row pass:    v = B_x S;  U = v exp(s(|v|^2));  S <- F_x U    (screen)
// B = swap F swap is the unnormalised inverse DFT.
//
// Row-oriented kernels hold the two rows of a unit as the two lanes of every
// value: an x-transform of length n on each lane.
//
// Column-oriented kernels hold one column, the even rows in one lane and the
// odd rows in the other (again exactly a unit).  The y-transform of length n
// is then two transforms of length n/2, one per lane, joined by one radix-2
// step across the lanes (decimation in time):
//   X[k] = E[k] + W_n^k O[k],  X[k + n/2] = E[k] - W_n^k O[k]   (k < n/2),
// which leaves the pair (X[k], X[k + n/2]) in one value.  The propagator
// multiplies it there, and the inverse starts with the mirror step
// (decimation in frequency) on the swapped values Y = swap(X P):
//   A[k] = Y[k] + Y[k + n/2],  B[k] = (Y[k] - Y[k + n/2]) W_n^k,
// whose two length-n/2 transforms return the even and odd output rows, i.e.
// the unit again.
#pragma once
#include <cuda.h>

#include "adjoint.cuh"
#include "pair.cuh"
#include "tma.cuh"

namespace nlse {

using pr::C2;
using pr::F2;

// ------------------------------------------------------------- geometry --

// Elements (pairs) per thread: E = 16 (radix-16 passes, 128 registers per
// thread, 512 threads per SM) or E = 8 (radix-8 passes, 64 registers, 1024
// threads per SM: twice the warps, one more exchange per transform); at most L.
template <int L, int E> __host__ __device__ constexpr int p_e() { return L < E ? L : E; }
template <int L, int E> __host__ __device__ constexpr int p_tpl() { return L / p_e<L, E>(); }
// row pairs per block of the row-oriented kernels: at least one warp.  A small
// grid is a few warps per SM whose serial chains bound the pass: blocks of one
// warp spread over all SMs (512^2, when introduced: 10.3 us per step with 32 threads
// per block, 11.0 with 128).
template <int N, int E> __host__ __device__ constexpr int p_rows() {
    return p_tpl<N, E>() >= 32 ? 1 : (32 / p_tpl<N, E>() > N / 2 ? N / 2 : 32 / p_tpl<N, E>());
}
template <int N, int E> __host__ __device__ constexpr int p_row_threads() { return p_tpl<N, E>() * p_rows<N, E>(); }
template <int N, int E> __host__ __device__ constexpr int p_row_smem() {
    return pr::pair_line_stride<N, p_e<N, E>(), p_rows<N, E>()>() * p_rows<N, E>() * 16;
}
// threads per column and shared memory of a C-column tile (sub-transform length n/2)
template <int N, int E> __host__ __device__ constexpr int p_col_tpl() { return p_tpl<N / 2, E>(); }
template <int N, int E, int C> __host__ __device__ constexpr int p_col_smem() {
    return pr::pair_line_stride<N / 2, p_e<N / 2, E>(), C>() * C * 16;
}
// resident blocks per SM for a budget of 128 (E = 16) or 64 (E = 8) registers
// per thread (a block narrower than a warp still takes a whole warp's registers)
template <int THREADS, int E> __host__ __device__ constexpr int p_min_blocks() {
    // blocks of two warps (1024^2: 3.4 of them per SM), and the radix-8 rows of the small
    // grids, run faster with all the registers a thread can have than with more of
    // them resident (1024^2 step 20.9 -> 19.2 us)
    constexpr int w = (THREADS + 31) / 32 * 32, budget = w == 64 || (E < 16 && w == 32) ? 256 : E >= 16 ? 512 : 1024;
    return w >= budget ? 1 : (budget / w > 32 ? 32 : budget / w);
}
// the same for the column kernels, whose radix-8 form needs about 85 registers
// per thread (the propagator and cross-lane factors on top of the transform)
template <int THREADS, int E> __host__ __device__ constexpr int p_col_min_blocks() {
    // blocks of one or two warps serve the small grids, which leave an SM a few of them:
    // no register limit (at 128 the transforms shorter than 512 points spilled; 256^2
    // step 8.8 -> 7.1 us, 512^2 10.3 -> 9.4, 1024^2 14.8 -> 14.6)
    constexpr int w = (THREADS + 31) / 32 * 32, budget = w <= 64 ? 256 : E >= 16 ? 512 : 768;
    return w >= budget ? 1 : (budget / w > 32 ? 32 : budget / w);
}

// Per-step FP32 twiddle block (one of kDither dithered copies, byte offsets
// from its start): the tables of the radix-16 march (pair.cuh: fused butterflies,
// 8-byte entries) for the n-point row transform and the n/2-point column
// sub-transforms, and those of the radix-8 march (radix-4 sub-passes) for the
// same.  After the last copy stand the tables of the one-off transforms, dithered
// as copy 0: the single-line table of fft.cuh (n entries of 8 bytes: lens,
// turbulence) and a radix-16 table of the row transform for the load prologue and
// the readouts (radix-4 sub-passes).
//
// Per-step propagator tables (one of kDitherP dithered copies): P_x, n entries
// of 8 bytes; P_y, n/2 pair entries of 16 bytes followed by the n/2 cross-lane
// factors W_n^k of the column pass (8 bytes each), all as (cos - 1, sin) of
// their angle (see col_body32).
//
// Why 256 copies (kDither): a few factors multiply most of the energy of a
// smooth beam every step -- the propagator and cross-lane factors of the low
// frequencies, and the pass-2 twiddles of the butterflies with k = 0 (the
// constants W_16^(i j) as table entries), which receive the low-frequency
// outputs of pass 1.  The residual error of a dithered factor over a cycle,
// up to 1/(2 kDither) of an FP32 unit, then changes the power coherently from
// cycle to cycle: with 16 copies the Kerr-only power drifted by 2e-6 over the
// 856 steps to the first collapse at 4096^2; with 256 (and P_x applied to each
// value, see col_body32) it stays within 1e-6.
constexpr int kDitherP = kDither;
__host__ __device__ constexpr size_t py32_copy_bytes(int n) { return (size_t)16 * (n / 2) + (size_t)8 * (n / 2); }
__host__ __device__ constexpr int tw32_min(int a, int b) { return a < b ? a : b; }
// Pair-table entry formats (pair.cuh): 8-byte (wx, wy), and 16-byte
// (wx, wx, wy, wy) for the radix-8 column transforms, whose kernel has no
// registers left for copies into both lanes.
using RowTab = float2;
template <int E> struct col_tab { using type = float2; };
template <> struct col_tab<8> { using type = float4; };
__host__ __device__ constexpr size_t tw32_row_off(int n, int e) {
    return e >= 16 ? 0 : (size_t)8 * (pr::fused_tab_entries(n, tw32_min(16, n)) +
                                      pr::fused_tab_entries(n / 2, tw32_min(16, n / 2)));
}
__host__ __device__ constexpr size_t tw32_col_off(int n, int e) {
    return e >= 16 ? tw32_row_off(n, 16) + (size_t)8 * pr::fused_tab_entries(n, tw32_min(16, n))
                   : (tw32_row_off(n, 8) + (size_t)8 * pr::pair_tab_entries(n, tw32_min(8, n)) + 15) / 16 * 16;
}
__host__ __device__ constexpr size_t tw32_copy_bytes(int n) {
    return (tw32_col_off(n, 8) + (size_t)16 * pr::pair_tab_entries(n / 2, tw32_min(8, n / 2)) + 255) / 256 * 256;
}
__host__ __device__ constexpr size_t tw32_line_off(int n) { return (size_t)kDither * tw32_copy_bytes(n); }
__host__ __device__ constexpr size_t tw32_oneoff_off(int n) { return tw32_line_off(n) + (size_t)8 * n; }
__host__ __device__ constexpr size_t tw32_region_bytes(int n) {
    return tw32_oneoff_off(n) + (size_t)8 * pr::pair_tab_entries(n, tw32_min(16, n));
}

// Global-memory access of the units: plain for the per-pass kernels, L2-only
// (.cg) for the persistent batched kernel whose fields other SMs rewrite.
struct UnitPlain {
    static constexpr bool kExactScreen = true;
    // read once per pass: no L1 allocation (the tables stay cached)
    __device__ __forceinline__ static C2 ld(const float4* p) {
        C2 v;
        asm volatile("ld.global.L1::no_allocate.v2.b64 {%0, %1}, [%2];" : "=l"(v.re.b), "=l"(v.im.b) : "l"(p));
        return v;
    }
    __device__ __forceinline__ static void st(float4* p, C2 v) {
        float4 f;
        pr::up(v.re, f.x, f.y);
        pr::up(v.im, f.z, f.w);
        *p = f;
    }
    __device__ __forceinline__ static void stores_next() { pdl_trigger(); }
};
struct UnitCG {
    static constexpr bool kExactScreen = false;
    __device__ __forceinline__ static C2 ld(const float4* p) {
        const float4 f = __ldcg(p);
        return {pr::pk(f.x, f.y), pr::pk(f.z, f.w)};
    }
    __device__ __forceinline__ static void st(float4* p, C2 v) {
        float4 f;
        pr::up(v.re, f.x, f.y);
        pr::up(v.im, f.z, f.w);
        __stcg(p, f);
    }
    __device__ __forceinline__ static void stores_next() {}
};

// --------------------------------------------------------------- screen --

namespace pr {

// the polynomials of kernels.cuh (expm1 to x^5, sin to x^9, cos - 1 to x^10),
// lane by lane, same operations in the same order
__device__ __forceinline__ F2 expm1_core2(F2 x) {
    F2 p = fma(x, bc(8.33333333333333333e-3f), bc(4.16666666666666667e-2f));
    p = fma(x, p, bc(1.66666666666666667e-1f));
    p = fma(x, p, bc(0.5f));
    return fma(mul(x, x), p, x);
}
__device__ __forceinline__ void sin_cosm1_core2(F2 r, F2& sr, F2& cr1) {
    const F2 r2 = mul(r, r);
    F2 ps = fma(r2, bc(2.75573192239858906e-6f), bc(-1.98412698412698413e-4f));
    ps = fma(r2, ps, bc(8.33333333333333333e-3f));
    ps = fma(r2, ps, bc(-1.66666666666666667e-1f));
    sr = fma(mul(r, r2), ps, r);
    F2 pc = fma(r2, bc(-2.75573192239858906e-7f), bc(2.48015873015873016e-5f));
    pc = fma(r2, pc, bc(-1.38888888888888889e-3f));
    pc = fma(r2, pc, bc(4.16666666666666667e-2f));
    pc = fma(r2, pc, bc(-0.5f));
    cr1 = mul(r2, pc);
}
// sin r to r^5 and cos r - 1 to r^6 (Taylor), for |r| <= 1/32
__device__ __forceinline__ void sin_cosm1_short2(F2 r, F2& sr, F2& cr1) {
    const F2 r2 = mul(r, r);
    const F2 ps = fma(r2, bc(8.33333333333333333e-3f), bc(-1.66666666666666667e-1f));
    sr = fma(mul(r, r2), ps, r);
    F2 pc = fma(r2, bc(-1.38888888888888889e-3f), bc(4.16666666666666667e-2f));
    pc = fma(r2, pc, bc(-0.5f));
    cr1 = mul(r2, pc);
}
__device__ __forceinline__ F2 ipow2(F2 u, int e) {
    F2 r = bc(1.0f), b = u;
#pragma unroll
    for (int bit = 0; bit < 5; ++bit) {  // K <= 16; e is uniform across the grid
        if (e & (1 << bit)) r = mul(r, b);
        b = mul(b, b);
    }
    return r;
}

// the general per-lane path of the screen (reduction of large phases, expf for
// large gains), kept out of line: it is rare, and inlined it would enlarge the
// row pass's instruction footprint
static __device__ __noinline__ void screen_slow2(float re0, float re1, float im0, float im1, int has_gain, unsigned warp,
                                          F2& em1, F2& sn, F2& cm1) {
    float s0, s1, k0, k1;
    sin_cosm1(im0, &s0, &k0, warp);
    sin_cosm1(im1, &s1, &k1, warp);
    em1 = has_gain ? pk(expm1_(re0, warp), expm1_(re1, warp)) : bc(0.0f);
    sn = pk(s0, s1);
    cm1 = pk(k0, k1);
}

// U = v + v d, d = exp(s(|v|^2)) - 1 = expm1(re) e^{i im} + (e^{i im} - 1), on both
// lanes: the per-step change, not the field, carries the rounding of the factor, and
// the whole of it is formed before a single rounding of v + v d (adding the small
// second-order part after the first would lose it at every step, coherently).
// Warp votes over both lanes of every thread pick a short polynomial (phases
// within 1/32 rad) or the full one (within pi/4); otherwise each lane takes
// the general scalar path of kernels.cuh.
__device__ __forceinline__ C2 apply_screen2(C2 v, const ScreenCoef<float>& c, unsigned warp) {
    const F2 u = mul(fma(v.re, v.re, mul(v.im, v.im)), bc(c.inv_iref));
    F2 uk1, uk;
    if (c.K == 8) {
        const F2 u2 = mul(u, u), u4 = mul(u2, u2);
        uk1 = mul(mul(u4, u2), u);
        uk = mul(u4, u4);
    } else {
        uk1 = ipow2(u, c.K - 1);
        uk = mul(uk1, u);
    }
    F2 re, im;
    if (c.real_gains) {  // (uniform) the zero terms of the general form, skipped: same values
        re = mul(bc(c.re_a), uk1);
        im = fma(bc(c.im_k), u, mul(bc(c.im_p), uk));
    } else {
        re = fma(bc(c.re_k), u, fma(bc(c.re_p), uk, mul(bc(c.re_a), uk1)));
        im = fma(bc(c.im_k), u, fma(bc(c.im_p), uk, mul(bc(c.im_a), uk1)));
    }
    float re0, re1, im0, im1;
    up(re, re0, re1);
    up(im, im0, im1);
    F2 em1, sn, cm1;
    const float ai = fmaxf(fabsf(im0), fabsf(im1)), ar = fmaxf(fabsf(re0), fabsf(re1));
    if (__all_sync(warp, ai <= 0.03125f && ar < 0.0625f)) {
        // phases within 1/32 rad (most of the field at most steps): sin to x^5
        // and cos - 1 to x^6, truncation below 1e-13 relative
        em1 = c.has_gain ? expm1_core2(re) : bc(0.0f);
        sin_cosm1_short2(im, sn, cm1);
    } else if (__all_sync(warp, ai <= 0.7853982f && ar < 0.0625f)) {
        em1 = c.has_gain ? expm1_core2(re) : bc(0.0f);
        sin_cosm1_core2(im, sn, cm1);
    } else {
        screen_slow2(re0, re1, im0, im1, c.has_gain, warp, em1, sn, cm1);
    }
    const F2 dre = fma(em1, cm1, add(em1, cm1));  // (1 + em1)(1 + cm1) - 1
    const F2 dim = fma(em1, sn, sn);              // (1 + em1) sin
    const F2 ddx = fma(v.re, dre, mul(v.im, neg(dim)));
    const F2 ddy = fma(v.re, dim, mul(v.im, dre));
    return {add(v.re, ddx), add(v.im, ddy)};
}

// The screen of all of a thread's values (apply_screens2).  The largest intensity
// of the warp's values bounds every phase and gain, so one vote picks the
// polynomials for all of them and the values follow each other without branches
// (a vote and two branches per value kept the sixteen dependent chains from
// overlapping).  K = 8 and real gains, the nominal case, have a short form: phases within 1/32 rad and
// gains below 2^-9 (expm1 to x^3, relative truncation below 4e-10; sin to x^5,
// cos - 1 to x^6, below 1e-13); middle form, for any K and gains: phases within
// pi/4, gains below 1/16; beyond, value by value (apply_screen2).
template <int FORM> __device__ __forceinline__ C2 screen_k8(C2 v, F2 u, const ScreenCoef<float>& c) {
    const F2 u2 = mul(u, u), u4 = mul(u2, u2);
    const F2 re = mul(bc(c.re_a), mul(mul(u4, u2), u));
    const F2 im = fma(bc(c.im_k), u, mul(bc(c.im_p), mul(u4, u4)));
    F2 em1, sn, cm1;
    if constexpr (FORM == 0) {
        em1 = fma(mul(re, re), fma(re, bc(1.66666666666666667e-1f), bc(0.5f)), re);
        sin_cosm1_short2(im, sn, cm1);
    } else {
        em1 = expm1_core2(re);
        sin_cosm1_core2(im, sn, cm1);
    }
    const F2 dre = fma(em1, cm1, add(em1, cm1));  // (1 + em1)(1 + cm1) - 1
    const F2 dim = fma(em1, sn, sn);              // (1 + em1) sin
    const F2 ddx = fma(v.re, dre, mul(v.im, neg(dim)));
    const F2 ddy = fma(v.re, dim, mul(v.im, dre));
    return {add(v.re, ddx), add(v.im, ddy)};
}
__device__ __forceinline__ F2 screen_u(C2 v, const ScreenCoef<float>& c) {
    return mul(fma(v.re, v.re, mul(v.im, v.im)), bc(c.inv_iref));
}
// The exact pointwise substep (kernels.cuh: apply_screen_exact) of all of a
// thread's values where the warp's largest absorption number |a| is at most 2^-7:
// amp - 1, f1 and fk by their power series to a^4 (truncation below 1e-10),
// U = v + v d as in the frozen screen; phases within 1/32 rad (FORM 0) or pi/4.
// The general form calls log1p, exp, three expm1 and sincos for every value.
template <int FORM> __device__ __forceinline__ C2 screen_exact2(C2 v, F2 u, const ScreenCoef<float>& c) {
    F2 uk1, uk;
    if (c.K == 8) {  // (uniform)
        const F2 u2 = mul(u, u), u4 = mul(u2, u2);
        uk1 = mul(mul(u4, u2), u);
        uk = mul(u4, u4);
    } else {
        uk1 = ipow2(u, c.K - 1);
        uk = mul(uk1, u);
    }
    const F2 a = mul(bc(c.ka), uk1), one = bc(1.0f);
    auto series = [&](const float (&k)[4]) {
        return mul(a, fma(a, fma(a, fma(a, bc(k[3]), bc(k[2])), bc(k[1])), bc(k[0])));
    };
    const F2 em1 = series(c.ex_amp), f1 = add(one, series(c.ex_f1)), fk = add(one, series(c.ex_fk));
    const F2 im = fma(mul(bc(c.im_k), u), f1, mul(mul(bc(c.im_p), uk), fk));
    F2 sn, cm1;
    if constexpr (FORM == 0) sin_cosm1_short2(im, sn, cm1);
    else sin_cosm1_core2(im, sn, cm1);
    const F2 dre = fma(em1, cm1, add(em1, cm1)), dim = fma(em1, sn, sn);
    const F2 ddx = fma(v.re, dre, mul(v.im, neg(dim))), ddy = fma(v.re, dim, mul(v.im, dre));
    return {add(v.re, ddx), add(v.im, ddy)};
}
__device__ __forceinline__ float ipow1(float u, int e) {
    float r = 1.0f;
    for (; e > 0; e >>= 1, u *= u)
        if (e & 1) r *= u;
    return r;
}
template <int E>
__device__ __forceinline__ void apply_screens_exact2(C2 (&v)[E], const ScreenCoef<float>& c, unsigned warp) {
    float um = 0.0f;
#pragma unroll
    for (int m = 0; m < E; ++m) {
        float u0, u1;
        up(screen_u(v[m], c), u0, u1);
        um = fmaxf(um, fmaxf(u0, u1));
    }
    const float p1 = ipow1(um, c.K - 1);
    const float phase = fabsf(c.im_k) * um + fabsf(c.im_p) * (p1 * um);  // f1, fk <= 1.01 at |a| <= 2^-7
    const bool series = fabsf(c.ka) * p1 <= 0.0078125f;
    if (__all_sync(warp, series && phase <= 0.0309f)) {
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = screen_exact2<0>(v[m], screen_u(v[m], c), c);
    } else if (__all_sync(warp, series && phase <= 0.7775f)) {
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = screen_exact2<1>(v[m], screen_u(v[m], c), c);
    } else {
#pragma unroll
        for (int m = 0; m < E; ++m) {
            float r0, r1, i0, i1;
            up(v[m].re, r0, r1);
            up(v[m].im, i0, i1);
            const float2 a = apply_screen_exact<float>(make_float2(r0, i0), c.inv_iref, c.im_k, c.im_p, c.ka, c.K);
            const float2 b = apply_screen_exact<float>(make_float2(r1, i1), c.inv_iref, c.im_k, c.im_p, c.ka, c.K);
            v[m] = {pk(a.x, b.x), pk(a.y, b.y)};
        }
    }
}
// exponent of the screen (kernels.cuh: screen_exponent) on both lanes, any K and gains
__device__ __forceinline__ void screen_exponent2(F2 u, const ScreenCoef<float>& c, F2& re, F2& im) {
    F2 uk1, uk;
    if (c.K == 8) {  // (uniform)
        const F2 u2 = mul(u, u), u4 = mul(u2, u2);
        uk1 = mul(mul(u4, u2), u);
        uk = mul(u4, u4);
    } else {
        uk1 = ipow2(u, c.K - 1);
        uk = mul(uk1, u);
    }
    re = fma(bc(c.re_k), u, fma(bc(c.re_p), uk, mul(bc(c.re_a), uk1)));
    im = fma(bc(c.im_k), u, fma(bc(c.im_p), uk, mul(bc(c.im_a), uk1)));
}
// (dre, dim) = e^{re + i im} - 1 by the middle form's polynomials
__device__ __forceinline__ void screen_delta2(F2 re, F2 im, F2& dre, F2& dim) {
    F2 sn, cm1;
    const F2 em1 = expm1_core2(re);
    sin_cosm1_core2(im, sn, cm1);
    dre = fma(em1, cm1, add(em1, cm1));
    dim = fma(em1, sn, sn);
}
template <int E> __device__ __forceinline__ void apply_screens2(C2 (&v)[E], const ScreenCoef<float>& c, unsigned warp) {
    float um = 0.0f;
#pragma unroll
    for (int m = 0; m < E; ++m) {
        float u0, u1;
        up(screen_u(v[m], c), u0, u1);
        um = fmaxf(um, fmaxf(u0, u1));
    }
    // (a NaN intensity is not seen by fmaxf: it goes through any form as NaN)
    if (c.K == 8 && c.real_gains) {  // (uniform)
        const float q2 = um * um, q4 = q2 * q2;
        const float gain = fabsf(c.re_a) * (q4 * q2 * um);
        const float phase = fabsf(c.im_k) * um + fabsf(c.im_p) * (q4 * q4);
        if (__all_sync(warp, phase <= 0.03125f && gain < 0.001953125f)) {
#pragma unroll
            for (int m = 0; m < E; ++m) v[m] = screen_k8<0>(v[m], screen_u(v[m], c), c);
            return;
        }
        if (__all_sync(warp, phase <= 0.7853982f && gain < 0.0625f)) {
#pragma unroll
            for (int m = 0; m < E; ++m) v[m] = screen_k8<1>(v[m], screen_u(v[m], c), c);
            return;
        }
    } else {
        const float p1 = ipow1(um, c.K - 1), pk = p1 * um;
        const float gain = fabsf(c.re_k) * um + fabsf(c.re_p) * pk + fabsf(c.re_a) * p1;
        const float phase = fabsf(c.im_k) * um + fabsf(c.im_p) * pk + fabsf(c.im_a) * p1;
        if (__all_sync(warp, phase <= 0.7853982f && gain < 0.0625f)) {
#pragma unroll
            for (int m = 0; m < E; ++m) {
                F2 re, im, dre, dim;
                screen_exponent2(screen_u(v[m], c), c, re, im);
                screen_delta2(re, im, dre, dim);
                v[m] = {add(v[m].re, fma(v[m].re, dre, mul(v[m].im, neg(dim)))),
                        add(v[m].im, fma(v[m].re, dim, mul(v[m].im, dre)))};
            }
            return;
        }
    }
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = apply_screen2(v[m], c, warp);
}

}  // namespace pr

// ------------------------------------------------------------- row tile --

// Screens of one row pair: v = the output of the inverse row transform (parts
// swapped) in, the field to transform forward out; with DIAG adds the thread's
// sum and max of |U|^2 (after the first screen); EXACT compiles the exact
// pointwise substep in.
template <bool DIAG, bool EXACT, int E>
__device__ __forceinline__ void row_screens32(C2 (&v)[E], const ScreenCoef<float>& sc, F2& fsum, float& tmax) {
    // the field entering the screen, swapped back
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = pr::swp(v[m]);
    if (sc.scale != 1.0f) {  // (uniform)
        const F2 s = pr::bc(sc.scale);
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = {pr::mul(v[m].re, s), pr::mul(v[m].im, s)};
    }
    const unsigned warp = (blockDim.x & 31) == 0 ? 0xffffffffu : __activemask();
#pragma unroll 1
    for (int rep = 0; rep < sc.reps; ++rep) {
        if (sc.active) {
            if (EXACT && sc.exact) {  // (uniform)
                pr::apply_screens_exact2(v, sc, warp);
            } else {
                pr::apply_screens2(v, sc, warp);
            }
        }
        if (DIAG && rep == 0) {
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const F2 a = pr::fma(v[m].re, v[m].re, pr::mul(v[m].im, v[m].im));
                fsum = pr::add(fsum, a);
                float a0, a1;
                pr::up(a, a0, a1);
                tmax = fmaxf(tmax, fmaxf(a0, a1));
            }
        }
    }
}

// Row pass transforms of one row pair held in v (B_x S swapped in): B_x,
// screen(s), F_x.  hook runs in the forward transform once the line is free
// (pair.cuh: fft_second).  Thread t holds the natural elements
// row_id<N, ER>(t) + m T.
template <int N, int ER> __device__ __forceinline__ int row_id(int t) {
    if constexpr (pr::mirrored(N, p_e<N, ER>())) return pr::nat_id<N>(t);
    else return t;
}
template <int N, int ER, bool DIAG, bool EXACT = true, class H = pr::NoHook>
__device__ __forceinline__ void row_body32(C2 (&v)[p_e<N, ER>()], C2* sm, const RowTab* __restrict__ tab,
                                           const ScreenCoef<float>& sc, int t, float& tsum, float& tmax,
                                           const H& hook = H{}) {
    constexpr int E = p_e<N, ER>();
    using S = pr::LineSync<p_tpl<N, ER>()>;
    F2 fsum = pr::bc(0.0f);
    if constexpr (pr::mirrored(N, E)) {
        pr::fft_first<N, S>(v, sm, tab, t);
        row_screens32<DIAG, EXACT>(v, sc, fsum, tmax);
        pr::fft_second<N, S, 1>(v, sm, tab, t, hook);
    } else {
        static_assert(H::none, "the hook is for the mirrored transforms");
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            pr::fft_pair<N, E, S, (ER >= 16)>(v, sm, tab, t);
            if (half == 0) row_screens32<DIAG, EXACT>(v, sc, fsum, tmax);
        }
    }
    if (DIAG) tsum += pr::lo(fsum) + pr::hi(fsum);
}

// Row pass body for the row pairs pair0 .. pair0 + p_rows - 1 (group g of
// p_tpl threads per pair): v = B_x S, screen(s), S = F_x U; with DIAG adds
// the thread's sum and max of |U|^2 (after the first screen).
template <int N, int ER, int RP, bool DIAG, class M>
__device__ __forceinline__ void row_tile32(const float4* src, float4* dst, const unsigned char* twb,
                                           const ScreenCoef<float>& sc, int pair0, C2* smem, float& tsum,
                                           float& tmax) {
    constexpr int E = p_e<N, ER>(), T = p_tpl<N, ER>();
    constexpr int LS = pr::pair_line_stride<N, E, RP>();
    const int g = (int)threadIdx.x / T, t = (int)threadIdx.x % T, j = row_id<N, ER>(t);
    const size_t row = (size_t)(pair0 + g) * N;
    C2* sm = smem + g * LS;
    const RowTab* tab = reinterpret_cast<const RowTab*>(twb + tw32_row_off(N, ER));
    C2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = pr::swp(M::ld(src + row + j + m * T));  // B_x = swap F_x swap
    row_body32<N, ER, DIAG, M::kExactScreen>(v, sm, tab, sc, t, tsum, tmax);
    M::stores_next();
#pragma unroll
    for (int m = 0; m < E; ++m) M::st(dst + row + j + m * T, v[m]);
}

// ---------------------------------------------------------- column body --

// Factors near 1.  The cross-lane factors W_n^k and the propagator factors
// P_x(k), P_y(k) = e^{i phi} are held as (d, s) = (cos phi - 1, sin phi) and
// applied as x + x (d + i s): the same two fused operations per part as a
// plain product, but the stored numbers are small where phi is small -- the
// low frequencies that carry most of a smooth beam's energy -- so their
// (dithered) rounding, and with it the residual magnitude error that would
// add up coherently over the steps, is relative to d and s, not to 1.
__device__ __forceinline__ void cmul_1d(float xr, float xi, float2 w, float& re, float& im) {
    re = fmaf(xr, w.x, fmaf(xi, -w.y, xr));
    im = fmaf(xi, w.x, fmaf(xr, w.y, xi));
}

// Column transform body: v holds units (t + m T, col) of one column (lanes:
// even and odd rows); computes B_y(P_x(col) rot P_y / n^2 F_y .) and leaves
// the output units in v.  tw: the step's twiddle block; px: n entries (d, s)
// of P_x; py: n/2 entries (d[k], d[k+n/2], s[k], s[k+n/2]) of P_y (without
// its 1/n^2, which goes with P_x: a power of two, exact), then the n/2
// cross-lane factors (d, s), both with entry k at col_pos(n/2, k).
template <int L> __device__ __forceinline__ void col_middle32(C2& v, int pos, const float2* __restrict__ cross,
                                                              const float4* __restrict__ py, F2 qx, F2 qy, F2 nqy,
                                                              F2 xd, F2 xs, F2 nxs) {
    const float2 w = pr::ld1(cross + pos);  // (cos - 1, sin) of W_n^k
    // X[k] = E + t, X[k + L] = E - t, t = W_n^k O
    float er, orr, ei, oi;
    pr::up(v.re, er, orr);
    pr::up(v.im, ei, oi);
    float tr, ti;
    cmul_1d(orr, oi, w, tr, ti);
    C2 X = {pr::pk(er + tr, er - tr), pr::pk(ei + ti, ei - ti)};
    // rot / n^2 and P_x (both lanes), then P_y (per lane): X + X (d + i s)
    X = pr::cmulw(X, qx, qy, nqy);
    X = {pr::fma(X.re, xd, pr::fma(X.im, nxs, X.re)), pr::fma(X.im, xd, pr::fma(X.re, xs, X.im))};
    F2 yd, ys;
    pr::ld_lanes(py + pos, yd, ys);
    X = {pr::fma(X.re, yd, pr::fma(X.im, pr::neg(ys), X.re)), pr::fma(X.im, yd, pr::fma(X.re, ys, X.im))};
    // Y = swap(X): A = Y[k] + Y[k + L], B = (Y[k] - Y[k + L]) W_n^k
    float yr0, yr1, yi0, yi1;
    pr::up(X.im, yr0, yr1);
    pr::up(X.re, yi0, yi1);
    float br, bi;
    cmul_1d(yr0 - yr1, yi0 - yi1, w, br, bi);
    v = {pr::pk(yr0 + yr1, br), pr::pk(yi0 + yi1, bi)};
}
template <int N, int EC, class S, int IL = 1>
__device__ __forceinline__ void col_body32(C2 (&v)[p_e<N / 2, EC>()], C2* sm, const unsigned char* twb,
                                           const float2* __restrict__ px, const float4* __restrict__ py,
                                           float2 rot, int col, int t) {
    constexpr int L = N / 2, E = p_e<L, EC>(), T = p_tpl<L, EC>();
    const auto* tab = reinterpret_cast<const typename col_tab<EC>::type*>(twb + tw32_col_off(N, EC));
    const float2* cross = reinterpret_cast<const float2*>(py + L);  // after the n/2 P_y entries
    auto middle = [&](int k0) {  // elements k0 + m T
        // rot / n^2 (a power of two: exact) and P_x(col) = 1 + d + i s, each
        // applied to every value (their product, rounded once per column,
        // would carry a magnitude error common to the column's values)
        constexpr float inv_n2 = 1.0f / ((float)N * (float)N);
        const F2 qx = pr::bc(rot.x * inv_n2), qy = pr::bc(rot.y * inv_n2), nqy = pr::bc(-rot.y * inv_n2);
        const float2 pxd = pr::ld1(px + col);
        const F2 xd = pr::bc(pxd.x), xs = pr::bc(pxd.y), nxs = pr::bc(-pxd.y);
        const int p0 = pr::col_pos(L, k0);  // (permutes runs of L/16 entries, and T is a multiple of L/16)
#pragma unroll
        for (int m = 0; m < E; ++m) col_middle32<L>(v[m], p0 + m * T, cross, py, qx, qy, nqy, xd, xs, nxs);
    };
    if constexpr (pr::mirrored(L, E)) {
        pr::fft_first<L, S, IL>(v, sm, tab, t);
        middle(pr::mid_id<L>(t));
        pr::fft_second<L, S, IL>(v, sm, tab, t);
    } else {
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            pr::fft_pair<L, E, S, (EC >= 16), IL>(v, sm, tab, t);
            if (half == 0) middle(t);
        }
    }
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = pr::swp(v[m]);  // B_y = swap F swap
}

// ---------------------------------------------------------------- kernels --

// Row pass of the march; with DIAG the block also reduces sum |U|^2 and
// max |U|^2 of its rows into partials.  At 4096^2: 98.9 -> 84.5 us (mirrored
// transforms with fused butterflies, one vote for the screens of a thread).  HBM
// (40 us at the copy bandwidth), the FMA pipe and the L1 data path are each about
// half busy: two blocks of eight warps per SM, all that 128 registers per thread
// allow, overlap each other's phases only in part (three blocks at 80 registers spill:
// 103 us; persistent blocks fetching the next row pair, k_row_pass32_pf: 90 us).
template <int N, int ER, bool DIAG>
__global__ void __launch_bounds__(p_row_threads<N, ER>(), p_min_blocks<p_row_threads<N, ER>(), ER>())
k_row_pass32(const float4* src, float4* dst, const unsigned char* twb, ScreenCoef<float> sc,
             double* __restrict__ partials) {
    extern __shared__ __align__(16) unsigned char smraw[];
    float tsum = 0.0f, tmax = 0.0f;
    pdl_wait();
    row_tile32<N, ER, p_rows<N, ER>(), DIAG, UnitPlain>(src, dst, twb, sc, blockIdx.x * p_rows<N, ER>(),
                                                         reinterpret_cast<C2*>(smraw), tsum, tmax);
    if constexpr (DIAG) block_partials<float>(tsum, tmax, partials);
}

// hook of fft_second that does something
template <class F> struct LineFree {
    static constexpr bool none = false;
    const F& f;
    __device__ __forceinline__ void operator()() const { f(); }
};

// One contiguous bulk copy of `bytes` (a multiple of 16; both addresses 16-byte
// aligned) from global into shared memory, counted in bytes on bar.
__device__ __forceinline__ void bulk_load_1d(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// block_partials<float> (kernels.cuh) for partial slot `slot`, usable again by
// the same block: the same reduction order, so the same bits.
__device__ __forceinline__ void block_partials32_at(float tsum, float tmax, double* __restrict__ partials, int slot) {
    __shared__ float red_s[32];
    __shared__ float red_m[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        tsum += __shfl_xor_sync(0xffffffffu, tsum, o);
        tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { red_s[warp] = tsum; red_m[warp] = tmax; }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = blockDim.x >> 5;
        float ss = 0.0f, mm = 0.0f;
        for (int w = 0; w < nw; ++w) { ss += red_s[w]; mm = fmaxf(mm, red_m[w]); }
        partials[2 * slot] = (double)ss;
        partials[2 * slot + 1] = (double)mm;
    }
    __syncthreads();  // red_s / red_m are free again
}

// Row pass with persistent blocks (one row pair per block at a time, n >= 2048
// at radix 16): block b takes row pairs b, b + G, b + 2G, ... (G blocks).  A
// row pair is n contiguous units; 16 bulk copies move its 16th parts to the
// starts of the line's regions (pair.cuh: Mirror), where each thread finds the
// elements it starts with in the slots it then writes first; the copies for
// the next row pair are issued as soon as the forward transform has read the
// line for the last time, and land while
// the last transform pass, the stores and the partials of the current row
// pair run.  Arithmetic, stores and partials (one slot per row pair) are those
// of k_row_pass32 at radix 16, bit for bit.  The wait for the copies is bounded
// as in the staged column pass (status bits 2 and 4, tma.cuh).  extra_tx (a test
// hook, 0 in use) makes block 0 expect that many bytes more for its first row
// pair than the copies bring, so that its wait runs out.
template <int N, bool DIAG>
__global__ void __launch_bounds__(p_tpl<N, 16>(), p_min_blocks<p_tpl<N, 16>(), 16>())
k_row_pass32_pf(const float4* src, float4* dst, const unsigned char* twb, ScreenCoef<float> sc,
                double* __restrict__ partials, int* __restrict__ status, uint32_t extra_tx) {
    constexpr int E = p_e<N, 16>(), T = p_tpl<N, 16>(), NP = N / 2;
    constexpr int RS = pr::Mirror<N>::RS;
    static_assert(p_rows<N, 16>() == 1 && T % 32 == 0, "one row pair of whole warps per block");
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ uint64_t bar;
    __shared__ int s_fail;
    C2* line = reinterpret_cast<C2*>(smraw);
    const RowTab* tab = reinterpret_cast<const RowTab*>(twb + tw32_row_off(N, 16));
    const int t = (int)threadIdx.x, j = pr::nat_id<N>(t);
    auto load_pair = [&](int p, uint32_t extra) {
        mbar_expect_tx(&bar, (uint32_t)N * 16 + extra);
#pragma unroll 1
        for (int r = 0; r < 16; ++r) bulk_load_1d(line + r * RS, src + (size_t)p * N + r * T, T * 16, &bar);
    };
    pdl_wait();
    if (threadIdx.x == 0) {
        s_fail = 0;
        mbar_init(&bar, 1);
        if ((int)blockIdx.x < NP) load_pair(blockIdx.x, blockIdx.x == 0 ? extra_tx : 0u);
    }
    __syncthreads();
    uint32_t parity = 0;
#pragma unroll 1
    for (int p = blockIdx.x; p < NP; p += gridDim.x) {
        if (threadIdx.x == 0 && !mbar_wait_bounded(&bar, parity)) {
            if (status) atomicOr(status, 2);
            // the copy still targets this block's memory: wait for it once more
            if (!mbar_wait_bounded(&bar, parity) && status) atomicOr(status, 4);
            s_fail = 1;
        }
        parity ^= 1u;
        __syncthreads();
        if (s_fail) return;  // (uniform)
        C2 v[E];
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = pr::swp(line[j + m * RS]);  // B_x = swap F_x swap
        const int next = p + (int)gridDim.x;
        float tsum = 0.0f, tmax = 0.0f;
        auto fetch_next = [&]() {
            if (threadIdx.x == 0 && next < NP) {
                fence_proxy_async_smem();  // the exchanges' accesses of the line, before the copies' writes
                load_pair(next, 0u);
            }
        };
        row_body32<N, 16, DIAG, true, LineFree<decltype(fetch_next)>>(v, line, tab, sc, t, tsum, tmax, {fetch_next});
        if (next >= NP) pdl_trigger();
#pragma unroll
        for (int m = 0; m < E; ++m) UnitPlain::st(dst + (size_t)p * N + j + m * T, v[m]);
        if constexpr (DIAG) block_partials32_at(tsum, tmax, partials, p);
    }
}

// Column tile with per-thread unit loads and stores: C columns from col0
// (column c = tid mod C: a warp's accesses cover C adjacent units per row pair).
template <int N, int EC, int C, class M>
__device__ __forceinline__ void col_tile32(const float4* src, float4* dst, const unsigned char* twb,
                                           const float2* __restrict__ px, const float4* __restrict__ py,
                                           float2 rot, int col0, C2* smem) {
    constexpr int L = N / 2, E = p_e<L, EC>(), T = p_tpl<L, EC>();
    constexpr int LS = pr::pair_line_stride<L, E, C>();
    const int c = (int)threadIdx.x % C, j = (int)threadIdx.x / C;
    const int col = col0 + c;
    C2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = M::ld(src + (size_t)(j + m * T) * N + col);
    col_body32<N, EC, pr::LineSync<T, C>>(v, smem + c * LS, twb, px, py, rot, col, j);
    M::stores_next();
#pragma unroll
    for (int m = 0; m < E; ++m) M::st(dst + (size_t)(j + m * T) * N + col, v[m]);
}

// Column pass, C columns per block with per-thread unit loads and stores.
template <int N, int EC, int C>
__global__ void __launch_bounds__(p_col_tpl<N, EC>() * C, p_col_min_blocks<p_col_tpl<N, EC>() * C, EC>())
k_col_pass32(const float4* src, float4* dst, const unsigned char* twb, const float2* __restrict__ px,
             const float4* __restrict__ py, float2 rot) {
    extern __shared__ __align__(16) unsigned char smraw[];
    pdl_wait();
    col_tile32<N, EC, C, UnitPlain>(src, dst, twb, px, py, rot, blockIdx.x * C, reinterpret_cast<C2*>(smraw));
}

// The staged column tile exists where a column is a whole number of 256-unit
// boxes and the lines fit the shared memory.
template <int N, int EC, int C> __host__ __device__ constexpr bool p_col_tma_valid() {
    return N % (2 * kTmaBoxRows) == 0 && p_col_tpl<N, EC>() * C <= 1024 &&
           p_col_smem<N, EC, C>() + kTmaAlignPad <= 232448;
}
// Columns staged side by side: pairs of columns share boxes of 32-byte rows and
// interleaved lines and threads (pair.cuh: IL) where the tile is an even number
// of columns.  A box row of one column is half a 32-byte sector, so single
// columns move every sector twice between L2 and the SM, and the copies are
// counted by rows.
template <int N, int EC, int C> __host__ __device__ constexpr int p_col_il() {
    return C % 2 == 0 && EC == 16 && p_col_tpl<N, EC>() >= 16 ? 2 : 1;
}
// Place of a staged column in its transform line: where the mirrored
// transforms' regions start on 128-byte boundaries (n/2 = 2048, 4096), one box
// of n/32 units per region, so that each thread finds its first elements in the
// slots it writes first and leaves its results in the slots it read last (no
// barrier between); else boxes of 256 units one after the other.
template <int N, int EC> __host__ __device__ constexpr bool p_col_in_regions() {
    return pr::mirrored(N / 2, p_e<N / 2, EC>()) && N >= 4096;
}
__host__ __device__ constexpr int p_col_box_rows(int n, int ec) { return ec == 16 && n >= 4096 ? n / 32 : kTmaBoxRows; }
template <int N, int EC> __host__ __device__ constexpr int p_col_box_stride() {
    return p_col_in_regions<N, EC>() ? pr::pair_padded_len<N / 2, 16>() / 16 : kTmaBoxRows;
}

// One staged column: thread t of its p_col_tpl threads reads units t + m T
// from the line, transforms them (col_body32, bit for bit as
// k_col_pass32) and writes them back.  Every access of the line by other
// threads is ordered before the caller's next barrier.
template <int N, int EC, int IL>
__device__ __forceinline__ void col_line32(C2* line, const unsigned char* twb, const float2* __restrict__ px,
                                           const float4* __restrict__ py, float2 rot, int col, int t) {
    constexpr int L = N / 2, E = p_e<L, EC>(), T = p_tpl<L, EC>();
    constexpr bool REG = p_col_in_regions<N, EC>();
    constexpr int ST = (REG ? p_col_box_stride<N, EC>() : T) * IL;
    static_assert(!REG || p_col_box_rows(N, EC) == T, "one box per region");
    using S = pr::LineSync<T, IL>;
    C2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = line[t * IL + m * ST];
    if constexpr (!REG) S::all();  // the staged column is consumed; the transforms reuse its memory
    col_body32<N, EC, S, IL>(v, line, twb, px, py, rot, col, t);
    if constexpr (!REG && pr::mirrored(L, E)) S::all();  // the last exchange is read
#pragma unroll
    for (int m = 0; m < E; ++m) line[t * IL + m * ST] = v[m];
}
// the tile's columns col0 .. col0 + C - 1 in smem, thread tid of the block
template <int N, int EC, int C>
__device__ __forceinline__ void col_lines32(C2* smem, const unsigned char* twb, const float2* __restrict__ px,
                                            const float4* __restrict__ py, float2 rot, int col0, int tid) {
    constexpr int L = N / 2, T = p_tpl<L, EC>(), IL = p_col_il<N, EC, C>();
    constexpr int LS = pr::pair_line_stride<L, p_e<L, EC>(), C>();
    const int grp = tid / (T * IL), c = tid % IL, t = tid % (T * IL) / IL;
    col_line32<N, EC, IL>(smem + grp * LS * IL + c, twb, px, py, rot, col0 + grp * IL + c, t);
}
template <int N, int EC, int C>
__device__ __forceinline__ void col_stage_load(C2* smem, const CUtensorMap* map, int col0, uint64_t* bar) {
    constexpr int L = N / 2, IL = p_col_il<N, EC, C>(), LS = pr::pair_line_stride<L, p_e<L, EC>(), C>() * IL;
    constexpr int BR = p_col_box_rows(N, EC), BS = p_col_box_stride<N, EC>() * IL;
#pragma unroll 1
    for (int c = 0; c < C / IL; ++c)
#pragma unroll 1
        for (int b = 0; b < L / BR; ++b) tma_load_3d(smem + c * LS + b * BS, map, 4 * (col0 + c * IL), b * BR, 0, bar);
}
template <int N, int EC, int C>
__device__ __forceinline__ void col_stage_store(const C2* smem, const CUtensorMap* map, int col0) {
    constexpr int L = N / 2, IL = p_col_il<N, EC, C>(), LS = pr::pair_line_stride<L, p_e<L, EC>(), C>() * IL;
    constexpr int BR = p_col_box_rows(N, EC), BS = p_col_box_stride<N, EC>() * IL;
#pragma unroll 1
    for (int c = 0; c < C / IL; ++c)
#pragma unroll 1
        for (int b = 0; b < L / BR; ++b) tma_store_3d(map, 4 * (col0 + c * IL), b * BR, 0, smem + c * LS + b * BS);
}

// Column pass with the tile staged by bulk tensor copies: the columns land in
// their transform lines (the tensor maps describe the state as n/2 row pairs x
// 4 n words), are transformed there (col_line32), and one thread stores
// the lines with bulk tensor copies.  At 4096^2 90.3 -> 84 us, 2048^2 34.7 -> 27.4: the
// L1 data path (exchanges, staging, tables) is 65 % busy, HBM half, and a block waits
// a quarter of its time for its tile (per-thread loads of the same pairs: 113 us;
// per-thread stores: 105; three blocks per SM leave the tables no L1: 113).  Waits
// are bounded as in k_col_pass_tma (tma.cuh), with the same status bits.
template <int N, int EC, int C>
__global__ void __launch_bounds__(p_col_tpl<N, EC>() * C, p_col_min_blocks<p_col_tpl<N, EC>() * C, EC>())
k_col_pass32_tma(const __grid_constant__ CUtensorMap mload, const __grid_constant__ CUtensorMap mstore,
                 const unsigned char* twb, const float2* __restrict__ px, const float4* __restrict__ py, float2 rot,
                 int* __restrict__ status, uint32_t extra_tx) {
    constexpr uint32_t BYTES = (uint32_t)(C * (N / 2) * 16);
    static_assert(p_col_tma_valid<N, EC, C>(), "staged column tile");
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ uint64_t bar;
    __shared__ int s_fail;
    const uint32_t pad = (kTmaAlign - (smem_u32(smraw) & (kTmaAlign - 1))) & (kTmaAlign - 1);
    C2* smem = reinterpret_cast<C2*>(smraw + pad);
    const int col0 = blockIdx.x * C;
    pdl_wait();
    if (threadIdx.x == 0) {
        s_fail = 0;
        mbar_init(&bar, 1);
        mbar_expect_tx(&bar, BYTES + (blockIdx.x == 0 ? extra_tx : 0u));
        col_stage_load<N, EC, C>(smem, &mload, col0, &bar);
        if (!mbar_wait_bounded(&bar, 0)) {
            if (status) atomicOr(status, 2);
            // the copies still target this block's memory: wait for them once more
            if (!mbar_wait_bounded(&bar, 0) && status) atomicOr(status, 4);
            s_fail = 1;
        }
    }
    __syncthreads();
    if (s_fail) return;  // (uniform)
    col_lines32<N, EC, C>(smem, twb, px, py, rot, col0, threadIdx.x);
    pdl_trigger();
    fence_proxy_async_smem();
    __syncthreads();
    if (threadIdx.x == 0) {
        col_stage_store<N, EC, C>(smem, &mstore, col0);
        tma_store_commit_and_wait_read();
    }
}

// Forward row transform S = F_x U (load prologue): src row-major complex64,
// dst in the unit layout (a different buffer).
template <int N>
__global__ void __launch_bounds__(p_row_threads<N, 16>(), p_min_blocks<p_row_threads<N, 16>(), 16>())
k_row_forward32(const float2* __restrict__ src, float4* __restrict__ dst, const unsigned char* twb) {
    constexpr int E = p_e<N, 16>(), T = p_tpl<N, 16>(), RP = p_rows<N, 16>();
    constexpr int LS = pr::pair_line_stride<N, E, RP>();
    extern __shared__ __align__(16) unsigned char smraw[];
    const int g = (int)threadIdx.x / T, j = (int)threadIdx.x % T;
    const size_t p = (size_t)blockIdx.x * RP + g;
    const RowTab* tab = reinterpret_cast<const RowTab*>(twb + tw32_oneoff_off(N));
    C2 v[E];
    pdl_wait();
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const float2 a = src[(2 * p) * N + j + m * T], b = src[(2 * p + 1) * N + j + m * T];
        v[m] = {pr::pk(a.x, b.x), pr::pk(a.y, b.y)};
    }
    pr::fft_pair<N, E, pr::LineSync<T>, false>(v, reinterpret_cast<C2*>(smraw) + g * LS, tab, j);
    pdl_trigger();
#pragma unroll
    for (int m = 0; m < E; ++m) UnitPlain::st(dst + p * N + j + m * T, v[m]);
}

// Readout: U = B_x S / n per row pair (S in the unit layout); reduces sum/max
// |U|^2 into partials and optionally writes U times unrot (field_out) and
// |U|^2 (flu_out), row-major.
template <int N>
__global__ void __launch_bounds__(p_row_threads<N, 16>(), p_min_blocks<p_row_threads<N, 16>(), 16>())
k_readout32(const float4* __restrict__ state, const unsigned char* twb, float2* __restrict__ field_out,
            float* __restrict__ flu_out, double* __restrict__ partials, float2 unrot) {
    constexpr int E = p_e<N, 16>(), T = p_tpl<N, 16>(), RP = p_rows<N, 16>();
    constexpr int LS = pr::pair_line_stride<N, E, RP>();
    extern __shared__ __align__(16) unsigned char smraw[];
    const int g = (int)threadIdx.x / T, j = (int)threadIdx.x % T;
    const size_t p = (size_t)blockIdx.x * RP + g;
    const RowTab* tab = reinterpret_cast<const RowTab*>(twb + tw32_oneoff_off(N));
    C2 v[E];
    pdl_wait();
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = pr::swp(UnitPlain::ld(state + p * N + j + m * T));
    pr::fft_pair<N, E, pr::LineSync<T>, false>(v, reinterpret_cast<C2*>(smraw) + g * LS, tab, j);
    pdl_trigger();
    const float inv = 1.0f / (float)N;
    float tsum = 0.0f, tmax = 0.0f;
#pragma unroll
    for (int m = 0; m < E; ++m) {
        float r0, r1, i0, i1;
        pr::up(v[m].im, r0, r1);  // swapped back
        pr::up(v[m].re, i0, i1);
        const float2 u[2] = {make_float2(r0 * inv, i0 * inv), make_float2(r1 * inv, i1 * inv)};
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const float a = u[l].x * u[l].x + u[l].y * u[l].y;
            tsum += a;
            tmax = fmaxf(tmax, a);
            const size_t o = (2 * p + l) * N + j + m * T;
            if (field_out)
                field_out[o] = make_float2(u[l].x * unrot.x - u[l].y * unrot.y, u[l].x * unrot.y + u[l].y * unrot.x);
            if (flu_out) flu_out[o] = a;
        }
    }
    block_partials<float>(tsum, tmax, partials);
}

// ------------------------------------------------------ adjoint (FP32) --
//
// The backward sweep re-marches a segment and then needs, at every step, the
// field v = B_x T entering the step's screen (adjoint.cuh).  The re-march computes
// it anyway: its row pass (k_row_stash32) writes v over the stored T, in the order
// its threads hold it (thread t's element m at t + m T_row: contiguous across a
// warp, no matter which point it is), and the backward row pass (k_adj_row32) reads
// it back in the same order, so that it runs two transforms instead of three, on
// the pair engine's mirrored pair of transforms.

// Row pass of the re-march: v = B_x seg into seg (stash order), then, unless dst
// is null (the last step of a segment), the screen and dst = F_x U as
// k_row_pass32 gives it, bit for bit.  24 bytes per point: at 8192^2 409 us, as long
// as the row pass without the stash.
template <int N, int ER>
__global__ void __launch_bounds__(p_row_threads<N, ER>(), p_min_blocks<p_row_threads<N, ER>(), ER>())
k_row_stash32(float4* seg, float4* dst, const unsigned char* twb, ScreenCoef<float> sc) {
    constexpr int E = p_e<N, ER>(), T = p_tpl<N, ER>(), RP = p_rows<N, ER>();
    constexpr int LS = pr::pair_line_stride<N, E, RP>();
    using S = pr::LineSync<T>;
    extern __shared__ __align__(16) unsigned char smraw[];
    pdl_wait();
    const int g = (int)threadIdx.x / T, t = (int)threadIdx.x % T, j = row_id<N, ER>(t);
    const size_t row = ((size_t)blockIdx.x * RP + g) * N;
    C2* sm = reinterpret_cast<C2*>(smraw) + g * LS;
    const RowTab* tab = reinterpret_cast<const RowTab*>(twb + tw32_row_off(N, ER));
    const unsigned warp = (blockDim.x & 31) == 0 ? 0xffffffffu : __activemask();
    C2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = pr::swp(UnitPlain::ld(seg + row + j + m * T));
    auto screen = [&]() {
#pragma unroll
        for (int m = 0; m < E; ++m) {
            v[m] = pr::swp(v[m]);
            UnitPlain::st(seg + row + t + m * T, v[m]);
        }
        if (dst && sc.active) pr::apply_screens2(v, sc, warp);
    };
    if constexpr (pr::mirrored(N, E)) {
        pr::fft_first<N, S>(v, sm, tab, t);
        screen();
        if (!dst) return;  // (uniform)
        pr::fft_second<N, S>(v, sm, tab, t);
    } else {
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            pr::fft_pair<N, E, S, (ER >= 16)>(v, sm, tab, t);
            if (half == 0) {
                screen();
                if (!dst) return;  // (uniform)
            }
        }
    }
    pdl_trigger();
#pragma unroll
    for (int m = 0; m < E; ++m) UnitPlain::st(dst + row + j + m * T, v[m]);
}

// Pullback of the screen on one value of both lanes (adjoint.cuh): G = G_U in, G_v
// out; adds the six theta sums.
__device__ __forceinline__ C2 adj_value2(C2 v, C2 G, F2 u, F2 re, F2 im, F2 dre, F2 dim, const AdjCoef<float>& a,
                                         F2 (&th)[6]) {
    using namespace pr;
    const ScreenCoef<float>& c = a.sc;
    F2 k2, k1, k;
    if (c.K == 8) {  // (uniform)
        const F2 u2 = mul(u, u), u4 = mul(u2, u2);
        k2 = mul(u4, u2);
        k1 = mul(k2, u);
        k = mul(u4, u4);
    } else {
        k2 = c.K >= 2 ? ipow2(u, c.K - 2) : bc(0.0f);
        k1 = ipow2(u, c.K - 1);
        k = mul(k1, u);
    }
    const float Kf = (float)c.K, K1f = (float)(c.K - 1);
    const F2 sr = mul(fma(bc(K1f * c.re_a), k2, fma(bc(Kf * c.re_p), k1, bc(c.re_k))), bc(c.inv_iref));
    const F2 si = mul(fma(bc(K1f * c.im_a), k2, fma(bc(Kf * c.im_p), k1, bc(c.im_k))), bc(c.inv_iref));
    // U' = v + v d, c = conj(G) U'
    const F2 wr = add(v.re, fma(v.re, dre, mul(v.im, neg(dim))));
    const F2 wi = add(v.im, fma(v.re, dim, mul(v.im, dre)));
    const F2 cr = fma(G.re, wr, mul(G.im, wi)), ci = fma(G.re, wi, mul(neg(G.im), wr));
    const F2 h = fma(cr, sr, mul(ci, neg(si)));  // Re(c s')
    const F2 q = add(h, h);
    const F2 tk = mul(bc(a.aK), u), tp = mul(bc(a.aP), k), ta = mul(bc(a.aA), k1);
    th[0] = fma(tk, ci, th[0]);
    th[1] = fma(tk, cr, th[1]);
    th[2] = fma(tp, ci, th[2]);
    th[3] = fma(tp, cr, th[3]);
    th[4] = fma(ta, cr, th[4]);
    th[5] = fma(ta, neg(ci), th[5]);
    // conj(e^s) G + q v
    return {fma(q, v.re, add(G.re, fma(dre, G.re, mul(dim, G.im)))),
            fma(q, v.im, add(G.im, fma(dre, G.im, mul(neg(dim), G.re))))};
}

// The FP32 sums of a pair's two rows joined in FP64, like all others.  volatile: issued
// here, between the transforms, where the slow FP64 pipe is idle and its latency passes
// behind the second one (joined with the block's sums at the end instead, where nothing
// overlaps with them at 8192^2, one block per SM: 606 -> 648 us per launch)
__device__ __forceinline__ double join_rows(F2 g) {
    double s;
    asm volatile("add.rn.f64 %0, %1, %2;" : "=d"(s) : "d"((double)pr::lo(g)), "d"((double)pr::hi(g)));
    return s;
}
// Six per-thread sums added into acc[block][6], in a fixed order: each warp takes sums
// 0..5 in turn, its lanes every 32nd thread's value, then a shuffle tree.  (A tree of
// FP64 shuffles in every warp is 30 FP64 additions per thread: at 8192^2 a fifth of the
// kernel.)
template <int THREADS>
__device__ __forceinline__ void block_accumulate6_rows(const double (&g)[6], double* __restrict__ acc) {
    __shared__ double red[6][THREADS];
#pragma unroll
    for (int q = 0; q < 6; ++q) red[q][threadIdx.x] = g[q];
    __syncthreads();
    if constexpr (THREADS >= 32) {
        for (int q = (int)threadIdx.x >> 5; q < 6; q += THREADS / 32) {
            double s = 0.0;
            for (int i = (int)threadIdx.x & 31; i < THREADS; i += 32) s += red[q][i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if ((threadIdx.x & 31) == 0) acc[6 * blockIdx.x + q] += s;
        }
    } else {
        for (int q = threadIdx.x; q < 6; q += THREADS) {
            double s = 0.0;
            for (int i = 0; i < THREADS; ++i) s += red[q][i];
            acc[6 * blockIdx.x + q] += s;
        }
    }
}

// Backward row pass of one step (adjoint.cuh: k_adj_row) on the unit layout:
// gam <- F_x( adjoint screen( B_x gam ; v ) ), v from the stash; natural != 0: the
// stash holds v in natural order (written by the radix-8 row pass).  24 bytes per
// point, two transforms and about 60 packed operations per pair: at 8192^2 1626 us
// with three transforms on the single-line engine -> 606; bound like the row pass by
// the overlap of its phases.
template <int N>
__global__ void __launch_bounds__(p_row_threads<N, 16>(), p_min_blocks<p_row_threads<N, 16>(), 16>())
k_adj_row32(float4* gam, const float4* stash, const unsigned char* twb, AdjCoef<float> ac, double* __restrict__ acc,
            int natural) {
    constexpr int E = p_e<N, 16>(), T = p_tpl<N, 16>(), RP = p_rows<N, 16>();
    constexpr int LS = pr::pair_line_stride<N, E, RP>();
    constexpr bool MIR = pr::mirrored(N, E);
    using S = pr::LineSync<T>;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int g = (int)threadIdx.x / T, t = (int)threadIdx.x % T, j = row_id<N, 16>(t);
    const size_t row = ((size_t)blockIdx.x * RP + g) * N;
    C2* sm = reinterpret_cast<C2*>(smraw) + g * LS;
    const RowTab* tab = reinterpret_cast<const RowTab*>(twb + tw32_row_off(N, 16));
    C2 v[E];
    pdl_wait();
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = pr::swp(UnitPlain::ld(gam + row + j + m * T));
    F2 th[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) th[q] = pr::bc(0.0f);
    double sum[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    auto pullback = [&]() {
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = pr::swp(v[m]);  // G_U = B_x G_S
        if (!ac.sc.active) return;  // (uniform)
        const ScreenCoef<float>& sc = ac.sc;
        const unsigned warp = (blockDim.x & 31) == 0 ? 0xffffffffu : __activemask();
        int at = t;
        if constexpr (MIR)
            if (natural) at = pr::mid_id<N>(t);
        const float4* sv = stash + row + at;
        constexpr int G = E < 4 ? E : 4;  // values whose forms are voted on together
#pragma unroll
        for (int m0 = 0; m0 < E; m0 += G) {
            C2 w[G];
            float um = 0.0f;
#pragma unroll
            for (int i = 0; i < G; ++i) w[i] = UnitPlain::ld(sv + (m0 + i) * T);
#pragma unroll
            for (int i = 0; i < G; ++i) {
                float u0, u1;
                pr::up(pr::screen_u(w[i], sc), u0, u1);
                um = fmaxf(um, fmaxf(u0, u1));
            }
            const float p1 = pr::ipow1(um, sc.K - 1), pk = p1 * um;
            const float gain = fabsf(sc.re_k) * um + fabsf(sc.re_p) * pk + fabsf(sc.re_a) * p1;
            const float phase = fabsf(sc.im_k) * um + fabsf(sc.im_p) * pk + fabsf(sc.im_a) * p1;
            const bool poly = __all_sync(warp, phase <= 0.7853982f && gain < 0.0625f);
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const F2 u = pr::screen_u(w[i], sc);
                F2 re, im, dre, dim;
                pr::screen_exponent2(u, sc, re, im);
                if (poly) {
                    pr::screen_delta2(re, im, dre, dim);
                } else {
                    float r0, r1, i0, i1;
                    pr::up(re, r0, r1);
                    pr::up(im, i0, i1);
                    F2 em1, sn, cm1;
                    pr::screen_slow2(r0, r1, i0, i1, sc.has_gain, warp, em1, sn, cm1);
                    dre = pr::fma(em1, cm1, pr::add(em1, cm1));
                    dim = pr::fma(em1, sn, sn);
                }
                v[m0 + i] = adj_value2(w[i], v[m0 + i], u, re, im, dre, dim, ac, th);
            }
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) sum[q] = join_rows(th[q]);
    };
    if constexpr (MIR) {
        pr::fft_first<N, S>(v, sm, tab, t);
        pullback();
        pr::fft_second<N, S>(v, sm, tab, t);
    } else {
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            pr::fft_pair<N, E, S, true>(v, sm, tab, t);
            if (half == 0) pullback();
        }
    }
    pdl_trigger();
#pragma unroll
    for (int m = 0; m < E; ++m) UnitPlain::st(gam + row + j + m * T, v[m]);
    block_accumulate6_rows<p_row_threads<N, 16>()>(sum, acc);
}

// Loss and seed (adjoint.cuh: k_loss_seed) on the unit layout, natural order (the
// target is row-major): the one-off transforms of the load and the readouts.  Five
// FP64 instructions per point bound it (630 us of 1105 at 8192^2; 1486 on the
// single-line engine).
template <int N>
__global__ void __launch_bounds__(p_row_threads<N, 16>(), p_min_blocks<p_row_threads<N, 16>(), 16>())
k_loss_seed32(const float4* __restrict__ state, float4* __restrict__ gam, const double* __restrict__ target,
              const unsigned char* twb, double seed_scale, double* __restrict__ partials) {
    constexpr int E = p_e<N, 16>(), T = p_tpl<N, 16>(), RP = p_rows<N, 16>();
    constexpr int LS = pr::pair_line_stride<N, E, RP>();
    extern __shared__ __align__(16) unsigned char smraw[];
    const int g = (int)threadIdx.x / T, j = (int)threadIdx.x % T;
    const size_t p = (size_t)blockIdx.x * RP + g;
    C2* sm = reinterpret_cast<C2*>(smraw) + g * LS;
    const RowTab* tab = reinterpret_cast<const RowTab*>(twb + tw32_oneoff_off(N));
    C2 v[E];
#pragma unroll
    for (int m = 0; m < E; ++m) v[m] = pr::swp(UnitPlain::ld(state + p * N + j + m * T));
    const float inv = 1.0f / (float)N;
    const double scale4 = 4.0 * seed_scale;
    double part = 0.0;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        pr::fft_pair<N, E, pr::LineSync<T>, false>(v, sm, tab, j);
        if (half == 0) {
            const F2 iv = pr::bc(inv);
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const F2 re = pr::mul(v[m].im, iv), im = pr::mul(v[m].re, iv);  // U, swapped back
                float f[2], w[2];
                pr::up(pr::fma(re, re, pr::mul(im, im)), f[0], f[1]);
#pragma unroll
                for (int l = 0; l < 2; ++l) {
                    const double d = (double)f[l] - target[(2 * p + l) * N + j + m * T];
                    part += d * d;
                    w[l] = (float)(d * scale4) * inv;  // 4 (F - D) / sum D^2, and the 1/n of G_S = F_x G_U / n
                }
                const F2 ww = pr::pk(w[0], w[1]);
                v[m] = {pr::mul(re, ww), pr::mul(im, ww)};
            }
        }
    }
#pragma unroll
    for (int m = 0; m < E; ++m) UnitPlain::st(gam + p * N + j + m * T, v[m]);
    block_partials<double>(part, 0.0, partials);
}

}  // namespace nlse
