// pair.cuh -- FP32 transform engine of the march that works on two lines at
// once (arXiv 2306.15678, Eq. 2: the diffraction operator is applied in
// Fourier space, the screen of Eq. 3 pointwise).
//
// Lanes.  Every value a thread holds is a pair: the same element of two lines
// that go through identical operations -- two adjacent rows (the row pass), or
// the even and the odd rows of one column (the column pass, see pass32.cuh).
// Real and imaginary parts are kept apart, (re0, re1) and (im0, im1), each in
// one 64-bit register pair, so that every add, subtract, multiply and fused
// multiply-add of the butterflies, twiddles and screen is one packed FP32x2
// instruction (add/sub/mul/fma.rn.f32x2) for both lines; each lane rounds
// exactly as the scalar instruction would.  Multiplying by +-i is a renaming
// of the two parts, and so is the inverse transform: with swap(re, im) =
// (im, re), conj(F(conj x)) = swap(F(swap x)), so the engine only ever runs
// the forward transform.
//
// State layout.  Unit u = (p n + x) of an n x n state array holds, as four
// floats, (re(2p, x), re(2p+1, x), im(2p, x), im(2p+1, x)): one 16-byte load
// gives one pair of the row pass (rows 2p, 2p+1 at x) and of the column pass
// (column x at rows 2p, 2p+1).
//
// Algorithm.  Stockham autosort, radix R = E (16) except a smaller final
// radix, thread j of T = L/E holding elements j + m T (m < E) of its pair of
// lines in natural order in and out.  Two forms of a radix-R pass of stride NS:
//  - radix4_pass (the radix-8 march, the load prologue and the readouts): radix
//    R1 = min(R, 4) with stride NS and twiddles W_{R1 NS}^{rA k}, then radix
//    R2 = R/R1 with stride R1 NS and twiddles W_{R NS}^{i (k + jA NS)} (k = b mod NS);
//    the pass (NS > 1) owns (R1-1) NS entries W_{R1 NS}^{rA k} at (rA-1) NS + k,
//    followed by (R2-1) R1 NS entries W_{R NS}^{i kB} at (i-1) R1 NS + kB, 8 bytes
//    (wx, wy) each or 16 bytes (wx, wx, wy, wy), by the table pointer's type;
//  - fused_pass (the radix-16 march): a radix-4 sub-pass, then radix-2 stages
//    whose products are fused with the sums (below).
// All twiddles come from the dithered tables (fft.cuh: step s reads copy
// s mod kDither), so no fixed rounded constant multiplies a large share of the
// values; only the first pass (NS = 1, radix4_pass in both forms, where the
// second factors are the constants W_R^{i jA} common to every butterfly)
// multiplies by exact constants held as unevaluated FP32 pairs (hi + lo).  Pass
// outputs go through one padded shared-memory exchange of 16-byte pairs per pass
// boundary.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "fft.cuh"

namespace nlse {
namespace pr {

// ------------------------------------------------------------ packed lanes --

struct F2 {
    unsigned long long b;
};

__device__ __forceinline__ F2 pk(float lo, float hi) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.b) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void up(F2 a, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a.b));
}
__device__ __forceinline__ float lo(F2 a) {
    float x, y;
    up(a, x, y);
    return x;
}
__device__ __forceinline__ float hi(F2 a) {
    float x, y;
    up(a, x, y);
    return y;
}
__device__ __forceinline__ F2 bc(float x) { return pk(x, x); }
__device__ __forceinline__ F2 add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
    return r;
}
__device__ __forceinline__ F2 sub(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
    return r;
}
__device__ __forceinline__ F2 mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.b) : "l"(a.b), "l"(b.b));
    return r;
}
// a * b + c, fused, lane by lane
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.b) : "l"(a.b), "l"(b.b), "l"(c.b));
    return r;
}
// -a, lane by lane: written as two scalar negations, which the assembler takes
// into the operands of the packed instruction that uses the result (an xor of
// the sign bits costs two integer instructions; the same holds for bc() below)
__device__ __forceinline__ F2 neg(F2 a) {
    F2 r;
    asm("{\n\t.reg .f32 x, y;\n\tmov.b64 {x, y}, %1;\n\tneg.f32 x, x;\n\tneg.f32 y, y;\n\t"
        "mov.b64 %0, {x, y};\n\t}" : "=l"(r.b) : "l"(a.b));
    return r;
}

// complex pair: (re0, re1), (im0, im1)
struct C2 {
    F2 re, im;
};
__device__ __forceinline__ C2 cadd(C2 a, C2 b) { return {add(a.re, b.re), add(a.im, b.im)}; }
__device__ __forceinline__ C2 csub(C2 a, C2 b) { return {sub(a.re, b.re), sub(a.im, b.im)}; }
// a * w for w = (wx + i wy) given as packed operands and nwy = -wy:
// re = ar wx - ai wy, im = ar wy + ai wx, each with its last add fused
__device__ __forceinline__ C2 cmulw(C2 a, F2 wx, F2 wy, F2 nwy) {
    return {fma(a.re, wx, mul(a.im, nwy)), fma(a.re, wy, mul(a.im, wx))};
}
// swap of the real and imaginary parts (a renaming)
__device__ __forceinline__ C2 swp(C2 a) { return {a.im, a.re}; }

// twiddle entry at a compile-time offset (in entries) from a per-pass base,
// through the read-only path, as the packed operands (wx, wx) and (wy, wy);
// volatile so that the loads stay where they are used (hoisted, they would
// hold registers through the passes)
template <int OFF> __device__ __forceinline__ void ldw(const float2* base, F2& wx, F2& wy) {
    float x, y;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2+%3];" : "=f"(x), "=f"(y) : "l"(base), "n"(OFF * 8));
    wx = bc(x);
    wy = bc(y);
}
template <int OFF> __device__ __forceinline__ void ldw(const float4* base, F2& wx, F2& wy) {
    asm volatile("ld.global.nc.v2.b64 {%0, %1}, [%2+%3];" : "=l"(wx.b), "=l"(wy.b) : "l"(base), "n"(OFF * 16));
}
// a 16-byte entry holding a different factor per lane, (x0, x1, y0, y1), as
// the packed operands (x0, x1) and (y0, y1)
__device__ __forceinline__ void ld_lanes(const float4* p, F2& x, F2& y) {
    asm volatile("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(x.b), "=l"(y.b) : "l"(p));
}
// one FP32 complex table entry (x, y) through the read-only path
__device__ __forceinline__ float2 ld1(const float2* p) {
    float2 r;
    asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "l"(p));
    return r;
}

// ----------------------------------------------------------- exact factors --

// x * c with c given in double: an unevaluated FP32 pair hi + lo
__device__ __forceinline__ F2 mulc(F2 x, double c) {
    const float h = (float)c, l = (float)(c - (double)(float)c);
    return fma(x, bc(h), mul(x, bc(l)));
}
// x * c + y * d with constants c, d (hi + lo each)
__device__ __forceinline__ F2 dotc(F2 x, double c, F2 y, double d) {
    const float ch = (float)c, cl = (float)(c - (double)(float)c);
    const float dh = (float)d, dl = (float)(d - (double)(float)d);
    return fma(x, bc(ch), fma(y, bc(dh), fma(x, bc(cl), mul(y, bc(dl)))));
}

// a * W_16^J (forward: W_16 = exp(-2 pi i / 16))
template <int J> __device__ __forceinline__ C2 w16(C2 a) {
    constexpr int j = J & 15;
    constexpr double c1 = 0.92387953251128675613, s1 = 0.38268343236508977173, r2 = 0.70710678118654752440;
    if constexpr (j == 0) {
        return a;
    } else if constexpr (j == 4) {  // -i
        return {a.im, neg(a.re)};
    } else if constexpr (j == 8) {
        return {neg(a.re), neg(a.im)};
    } else if constexpr (j == 12) {  // +i
        return {neg(a.im), a.re};
    } else if constexpr ((j & 1) == 0) {
        // W^j = r2 (cx - i sx), cx, sx = +-1: re = r2 (cx x + sx y), im = r2 (cx y - sx x)
        constexpr int cx = (j == 2 || j == 14) ? 1 : -1;
        constexpr int sx = (j == 2 || j == 6) ? 1 : -1;
        // x + y and y - x (or their negatives) carry the signs; the constant r2 or -r2
        const F2 s = add(a.re, a.im), d = sub(a.im, a.re);
        // re = r2 (cx x + sx y):  j = 2: s;  6: d;  10: -s;  14: -d
        // im = r2 (cx y - sx x):  j = 2: d;  6: -s; 10: -d;  14: s
        constexpr double re_c = (cx == sx) ? cx * r2 : sx * r2;  // coefficient of s (cx == sx) or d
        constexpr double im_c = (cx == sx) ? cx * r2 : -sx * r2;
        if constexpr (cx == sx) return {mulc(s, re_c), mulc(d, im_c)};
        else return {mulc(d, re_c), mulc(s, im_c)};
    } else {
        // W^j = c - i s: re = x c + y s, im = y c - x s
        constexpr double c = j == 1 ? c1 : j == 3 ? s1 : j == 5 ? -s1 : j == 7 ? -c1
                           : j == 9 ? -c1 : j == 11 ? -s1 : j == 13 ? s1 : c1;
        constexpr double s = j == 1 ? s1 : j == 3 ? c1 : j == 5 ? c1 : j == 7 ? s1
                           : j == 9 ? -s1 : j == 11 ? -c1 : j == 13 ? -c1 : -s1;
        return {dotc(a.re, c, a.im, s), dotc(a.im, c, a.re, -s)};
    }
}

// ---------------------------------------------------------------- DFT_R --

__device__ __forceinline__ void dft2(C2& a0, C2& a1) {
    const C2 t = a0;
    a0 = cadd(t, a1);
    a1 = csub(t, a1);
}
// forward DFT_4; the products by -i and +i are renamings folded into the adds
__device__ __forceinline__ void dft4(C2& a0, C2& a1, C2& a2, C2& a3) {
    const C2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), d = csub(a1, a3);
    a0 = cadd(t0, t2);
    a2 = csub(t0, t2);
    a1 = {add(t1.re, d.im), sub(t1.im, d.re)};  // t1 - i d
    a3 = {sub(t1.re, d.im), add(t1.im, d.re)};  // t1 + i d
}

// --------------------------------------------------------- Stockham passes --

__host__ __device__ constexpr int split1(int r) { return r >= 4 ? 4 : r; }
__host__ __device__ constexpr int split2(int r) { return r / split1(r); }
// table entries of the pass with radix r and stride ns (none for ns = 1)
__host__ __device__ constexpr int pass_entries(int r, int ns) {
    return ns > 1 ? (split1(r) - 1) * ns + (split2(r) - 1) * split1(r) * ns : 0;
}
// first table entry of the pass with stride ns of an l-point transform with
// e elements per thread; pair_tab_offset(l, e, l) is the size of the table
__host__ __device__ constexpr int pair_tab_offset(int l, int e, int ns) {
    int off = 0, cur = 1;
    while (cur < ns) {
        const int rem = l / cur;
        const int r = rem >= e ? e : rem;
        off += pass_entries(r, cur);
        cur *= r;
    }
    return off;
}
__host__ __device__ constexpr int pair_tab_entries(int l, int e) { return pair_tab_offset(l, e, l); }

// padded shared-memory line (16-byte pairs): one spare slot every E elements, or
// the 16 regions of the mirrored transforms (below)
template <int L, int E> __host__ __device__ constexpr int pair_padded_len() {
    return E != 16 || L < 512 || L == 8192 ? L + L / E : L == 512 ? 16 * 49 : L == 1024 ? 16 * 81 : 16 * (L / 16 + 16);
}
// stride between the lines a block holds: a multiple of 8 slots (128 bytes:
// bulk-tensor copies land at line starts), plus a skew between lines
template <int L, int E, int LINES> __host__ __device__ constexpr int pair_line_stride() {
    constexpr int pl = pair_padded_len<L, E>();
    constexpr int base = (pl + 7) / 8 * 8;
    return LINES > 1 ? base + 8 : base;
}

template <int I, int END, typename F> __device__ __forceinline__ void sfor(F&& f) {
    if constexpr (I < END) {
        f(std::integral_constant<int, I>{});
        sfor<I + 1, END>(f);
    }
}

struct NoHook {
    static constexpr bool none = true;
    __device__ __forceinline__ void operator()() const {}
};

// Barriers of a transform: all() orders the threads of a whole line, in() the
// 16 or 32 threads that share a group exchange (below).  A line of at most 32
// consecutive threads sits in one warp, and so does every exchange group of a
// line of consecutive threads; lines whose threads are interleaved (`STEP`
// lines side by side) keep to a warp while 16 STEP <= 32.
template <bool LINE_IN_WARP, bool GROUP_IN_WARP> struct Sync {
    __device__ __forceinline__ static void all() {
        if constexpr (LINE_IN_WARP) __syncwarp();
        else __syncthreads();
    }
    __device__ __forceinline__ static void in() {
        if constexpr (GROUP_IN_WARP) __syncwarp();
        else __syncthreads();
    }
};
// T threads per line, STEP lines interleaved thread by thread (1: none)
template <int T, int STEP = 1> using LineSync = Sync<(T * STEP <= 32), (16 * STEP <= 32)>;

// position of entry k within the NS entries of one factor of a pass with
// stride ns: bits 2-3 and 4-5 of k exchanged where the transform runs as two
// mirrored ones (below), ns >= 256.  One of the two transforms reads k
// consecutive across the lanes, the other k = g + 16 i (i across the lanes);
// in 4 x 4 tiles each touches 4 lines of 8-byte entries per load (2 would be the
// least; stored in order the second would touch 16).
__host__ __device__ constexpr bool mirrored(int l, int e) { return e == 16 && l >= 512 && l <= 8192; }
__host__ __device__ constexpr int tile_pos(int k) { return (k & ~0x3C) | ((k >> 2) & 0xC) | ((k & 0xC) << 2); }
__host__ __device__ constexpr int tab_pos(int l, int e, int ns, int k) {
    return mirrored(l, e) && ns >= 256 ? tile_pos(k) : k;
}

// One Stockham pass of stride NS on the registers of logical thread j: element
// m in, output m out (m = i + r B of butterfly i).  Radix-4 sub-passes.
template <int L, int E, int NS, class TE>
__device__ __forceinline__ void radix4_pass(C2 (&v)[E], const TE* __restrict__ tab, int j) {
    constexpr int REM = L / NS;
    constexpr int R = REM >= E ? E : REM;
    constexpr int T = L / E;
    constexpr int B = E / R;
    constexpr int R1 = split1(R), R2 = split2(R);
    static_assert(E % R == 0, "radix must divide the elements per thread");
    static_assert(R == 1 || R == 2 || R == 4 || R == 8 || R == 16, "radix");
    constexpr int TA = pair_tab_offset(L, E, NS);  // sub-pass A entries
    constexpr int TB = TA + (R1 - 1) * NS;         // sub-pass B entries
#pragma unroll
    for (int i = 0; i < B; ++i) {
        const int b = j + i * T;
        const int k = NS > 1 ? (b & (NS - 1)) : 0;
        C2 a[R];
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = v[i + r * B];
        // sub-pass A: radix R1 over rA on registers ip + R2 rA, for each ip < R2
        if constexpr (NS > 1 && R1 > 1) {
            const TE* ta = tab + TA + k;
            sfor<1, R1>([&](auto rc) {
                constexpr int rA = decltype(rc)::value;
                F2 wx, wy;
                ldw<(rA - 1) * NS>(ta, wx, wy);
                const F2 nwy = neg(wy);
#pragma unroll
                for (int ip = 0; ip < R2; ++ip) a[ip + R2 * rA] = cmulw(a[ip + R2 * rA], wx, wy, nwy);
            });
        }
#pragma unroll
        for (int ip = 0; ip < R2; ++ip) {
            if constexpr (R1 == 4) dft4(a[ip], a[ip + R2], a[ip + 2 * R2], a[ip + 3 * R2]);
            else if constexpr (R1 == 2) dft2(a[ip], a[ip + R2]);
        }
        // sub-pass B: radix R2 over ip on registers ip + R2 jA, for each jA < R1
        if constexpr (R2 > 1) {
            if constexpr (NS > 1) {
                const TE* tb = tab + TB + k;
                sfor<0, R1>([&](auto jc) {
                    constexpr int jA = decltype(jc)::value;
                    sfor<1, R2>([&](auto ic) {
                        constexpr int ip = decltype(ic)::value;
                        F2 wx, wy;
                        ldw<(ip - 1) * R1 * NS + jA * NS>(tb, wx, wy);
                        a[ip + R2 * jA] = cmulw(a[ip + R2 * jA], wx, wy, neg(wy));
                    });
                });
            } else {
                sfor<0, R1>([&](auto jc) {
                    constexpr int jA = decltype(jc)::value;
                    sfor<1, R2>([&](auto ic) {
                        constexpr int ip = decltype(ic)::value;
                        a[ip + R2 * jA] = w16<ip * jA * (16 / R)>(a[ip + R2 * jA]);
                    });
                });
            }
#pragma unroll
            for (int jA = 0; jA < R1; ++jA) {
                if constexpr (R2 == 4) dft4(a[R2 * jA], a[R2 * jA + 1], a[R2 * jA + 2], a[R2 * jA + 3]);
                else if constexpr (R2 == 2) dft2(a[R2 * jA], a[R2 * jA + 1]);
            }
        }
        // output r = jA + R1 q sits in slot q + R2 jA
#pragma unroll
        for (int r = 0; r < R; ++r) v[i + r * B] = a[(r / R1) + R2 * (r % R1)];
    }
}

// -------------------------------------------------------- fused butterflies --
//
// The march's radix-16 engine takes the pass of stride NS > 1 by decimation in
// time: a radix-4 sub-pass on inputs multiplied by w^4, w^8, w^12 (w = W_{NS R}^k),
// then radix-2 stages x = e + c o, y = e - c o with c = W_{NS 2^s}^{k + NS j}, stage
// s = 3 (j < 4) and 4 (j < 8).  With c = p (1 + i q) or p (q + i), q the smaller of
// its parts over the larger, a stage's product and both sums are three fused
// multiply-adds per part: u = o (1 + i q) or o (q + i), x = e + p u, y = e - p u, 6
// for 4 real numbers (separate products and sums: 8), each result with two
// roundings.  Which form is fixed by j: the angle of c lies in the j-th part of a
// quarter turn.  c for j + 2^(s-2) is -i c for j (a renaming), so a pass of radix 16
// (8, 4) reads 9 (5, 3) entries instead of the 15 (7, 3) of two radix-4
// (radix-2) sub-passes.  (2 e - x for y would save nothing more and carry x's
// errors: field errors 10-20 % larger.)
// Table of the pass: entry q of each k at q NS + tab_pos(k): W_{4 NS}^{(q+1) k} for
// q < 3 (radix 2: W_{2 NS}^k), then (p, q) of stage 3, j < 2, and stage 4, j < 4.

__host__ __device__ constexpr int fused_q(int r) { return r == 16 ? 9 : r == 8 ? 5 : r == 4 ? 3 : 1; }
__host__ __device__ constexpr int fused_entries(int r, int ns) { return ns > 1 ? fused_q(r) * ns : 0; }
__host__ __device__ constexpr int fused_tab_offset(int l, int e, int ns) {
    int off = 0, cur = 1;
    while (cur < ns) {
        const int rem = l / cur;
        const int r = rem >= e ? e : rem;
        off += fused_entries(r, cur);
        cur *= r;
    }
    return off;
}
__host__ __device__ constexpr int fused_tab_entries(int l, int e) { return fused_tab_offset(l, e, l); }

// the twiddles of one thread's butterflies of a pass
template <int L, int E, int NS> struct PassTw {
    static constexpr int R = L / NS >= E ? E : L / NS;
    static constexpr int B = E / R;
    static constexpr int Q = NS > 1 ? fused_q(R) : 0;  // entries per butterfly
    float2 w[B * Q > 0 ? B * Q : 1];
};
template <int L, int E, int NS>
__device__ __forceinline__ PassTw<L, E, NS> load_tw(const float2* __restrict__ tab, int j) {
    using P = PassTw<L, E, NS>;
    constexpr int T = L / E;
    P p;
    if constexpr (NS > 1) {
        sfor<0, P::B>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            const float2* base = tab + fused_tab_offset(L, E, NS) + tab_pos(L, E, NS, (j + i * T) & (NS - 1));
            sfor<0, P::Q>([&](auto qc) {
                constexpr int q = decltype(qc)::value;
                asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2+%3];"
                             : "=f"(p.w[i * P::Q + q].x), "=f"(p.w[i * P::Q + q].y) : "l"(base), "n"(q * NS * 8));
            });
        });
    }
    return p;
}
// x = e + c o, y = e - c o; c = p (1 + i q) or (SINE) p (q + i), times -i if TURN
template <bool SINE, bool TURN> __device__ __forceinline__ void fused_butterfly(C2& e, C2& o, float2 w) {
    const F2 p = bc(w.x), q = bc(w.y);
    C2 u;
    if constexpr (!SINE) u = {fma(o.im, neg(q), o.re), fma(o.re, q, o.im)};
    else u = {fma(o.re, q, neg(o.im)), fma(o.im, q, o.re)};
    if constexpr (!TURN) {
        o = {fma(u.re, neg(p), e.re), fma(u.im, neg(p), e.im)};
        e = {fma(u.re, p, e.re), fma(u.im, p, e.im)};
    } else {  // -i u = (u.im, -u.re)
        o = {fma(u.im, neg(p), e.re), fma(u.re, p, e.im)};
        e = {fma(u.im, p, e.re), fma(u.re, neg(p), e.im)};
    }
}
template <int L, int E, int NS>
__device__ __forceinline__ void fused_pass(C2 (&v)[E], const PassTw<L, E, NS>& tw) {
    using P = PassTw<L, E, NS>;
    constexpr int R = P::R, B = P::B, BITS = ilog2(R), R2 = R >= 4 ? R / 4 : 1;
#pragma unroll
    for (int i = 0; i < B; ++i) {
        C2 a[R];
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = v[i + r * B];
        // radix-4 sub-pass on slots ip + R2 rA (radix 2: one butterfly)
        sfor<1, (R >= 4 ? 4 : R)>([&](auto rc) {
            constexpr int rA = decltype(rc)::value;
            const float2 w = tw.w[i * P::Q + rA - 1];
            const F2 wx = bc(w.x), wy = bc(w.y), nwy = neg(wy);
#pragma unroll
            for (int ip = 0; ip < R2; ++ip) a[ip + R2 * rA] = cmulw(a[ip + R2 * rA], wx, wy, nwy);
        });
        if constexpr (R >= 4) {
#pragma unroll
            for (int ip = 0; ip < R2; ++ip) dft4(a[ip], a[ip + R2], a[ip + 2 * R2], a[ip + 3 * R2]);
        } else {
            dft2(a[0], a[1]);
        }
        // stage s: output j < 2^(s-1) of base r0 and of base r0 + R / 2^s
        // (slots: base + R2 (j mod 4), plus R / 8 from j = 4 on) make j and j + 2^(s-1)
        sfor<3, BITS + 1>([&](auto sc) {
            constexpr int s = decltype(sc)::value, half = 1 << (s - 1), step = R >> s, nq = half / 2;
            sfor<0, half>([&](auto jc) {
                constexpr int j = decltype(jc)::value, slot = R2 * (j % 4) + (j / 4) * (R / 8);
                const float2 w = tw.w[i * P::Q + (s == 3 ? 3 : 5) + j % nq];
#pragma unroll
                for (int r0 = 0; r0 < step; ++r0)
                    fused_butterfly<(j % nq >= nq / 2), (j >= nq)>(a[slot + r0], a[slot + step + r0], w);
            });
        });
        sfor<0, R>([&](auto jc) {
            constexpr int j = decltype(jc)::value;
            // radix 16: j + 8 at the slot of j plus 1; radix 8: j + 4 at the slot of j plus 1
            constexpr int slot = R == 16 ? 4 * (j % 4) + 2 * (j / 4 % 2) + j / 8 : R == 8 ? 2 * (j % 4) + j / 4 : j;
            v[i + j * B] = a[slot];
        });
    }
}

// Forward transform of a pair of lines of length L held in v (layout above),
// natural order in and out.  `sm` is this group's padded line
// (pair_padded_len<L, E>() slots); every thread of the line (of the block,
// where S::all() is the block's barrier) must call this.  FUSED: the
// butterflies above with their table (8-byte entries), else radix-4 sub-passes.
// IL: interleaved lines (below, Mirror).
template <int L, int E, class S, bool FUSED, int IL = 1, int NS = 1, class TE>
__device__ __forceinline__ void fft_pair(C2 (&v)[E], C2* sm, const TE* __restrict__ tab, int j) {
    constexpr int REM = L / NS;
    constexpr int R = REM >= E ? E : REM;
    constexpr int T = L / E;
    constexpr int B = E / R;
    if constexpr (NS == 1 || !FUSED) radix4_pass<L, E, NS>(v, tab, j);
    else fused_pass<L, E, NS>(v, load_tw<L, E, NS>(tab, j));
    if constexpr (NS * R < L) {
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const int b = j + i * T;
            const int base = ((b >> ilog2(NS)) << ilog2(NS * R)) + (NS > 1 ? (b & (NS - 1)) : 0);
#pragma unroll
            for (int r = 0; r < R; ++r) sm[padix<E>(base + r * NS) * IL] = v[i + r * B];
        }
        S::all();
#pragma unroll
        for (int m = 0; m < E; ++m) v[m] = sm[padix<E>(j + m * T) * IL];
        S::all();
        fft_pair<L, E, S, FUSED, IL, NS * R>(v, sm, tab, j);
    }
}

// ------------------------------------------------ two mirrored transforms --
//
// A pass of the march runs two transforms with a pointwise operation between
// them, so the order of the points in between is free.  The first transform
// (fft_first) starts from the natural order and ends with thread t holding the
// natural elements J + m T of another thread J = mid_id(t); the second
// (fft_second) starts there and ends in natural order.  Both are the Stockham
// passes above, with the same operations on the same values, done by other
// threads: after the first radix-16 pass of the first transform the line falls
// into 16 independent transforms of length L/16, each held by L/256 threads
// of one warp, so only the exchange before them crosses warps, and likewise
// only the last wide exchange of the second transform.  Two barriers across the
// line per pair of transforms, instead of two at each of four (L = 8192: six)
// exchanges: at 4096^2 the passes waited there in lockstep.
//
// Shared memory holds 16 regions of RS slots (region r: the sub-transform of
// output r).  Every exchange across warps is written to, or read from, slots
// that only the same thread used before (slot m RS + t for element t + m T),
// so no barrier is needed ahead of its writes; a group's exchanges stay within
// its own regions.  RS and the strides inside the regions keep every 8 lanes
// of a 16-byte access on different banks.

template <int L> struct Mirror {
    static constexpr int T = L / 16;           // threads per line
    static constexpr int TG = L / 256;         // threads per sub-transform: 2, 4, 8, 16, 32
    static constexpr int R3 = TG < 16 ? TG : 16;
    static constexpr int NG = 16 / R3;         // sub-transforms per group of 16 threads
    static constexpr int RS = L == 512 ? 49 : L == 1024 ? 81 : T + 16;
    static constexpr int LINE = 16 * RS;       // slots
};
// natural element of thread t in fft_first's input and fft_second's output
template <int L> __device__ __forceinline__ int nat_id(int t) {
    if constexpr (L == 8192) return (t & 15) + 16 * (t >> 5) + 256 * ((t >> 4) & 1);
    else return t;
}
// natural element of thread t between the two transforms
template <int L> __device__ __forceinline__ int mid_id(int t) {
    using G = Mirror<L>;
    if constexpr (L == 8192) return (t >> 5) + 16 * (t & 31);
    else return (t >> 4) + G::R3 * ((t & 15) / G::TG) + 16 * ((t & 15) % G::TG);
}

// Place of entry k of a column's P_y and cross-lane tables (l entries, read
// between the two transforms): within each run of T = l/16 entries, those that a
// warp reads together side by side, J = mid_id(t) for 32 consecutive t; pairs of
// neighbours stay together, so that readers in natural order (the radix-8
// passes) still use whole 32-byte sectors.
__host__ __device__ constexpr int col_pos(int l, int k) {
    if (!mirrored(l, 16) || l > 4096) return k;
    const int T = l / 16, R3 = l / 256, J = k % T;
    return (J & 1) + 2 * (J / R3) + 32 * ((J >> 1) % (R3 / 2)) + (k - J);
}

template <int L, class S, int IL = 1>
__device__ __forceinline__ void fft_first(C2 (&v)[16], C2* sm, const float2* __restrict__ tab, int t) {
    using G = Mirror<L>;
    constexpr int RS = G::RS * IL, TG = G::TG * IL, TP = TG + IL;  // in units of the interleaved line
    radix4_pass<L, 16, 1>(v, tab, t);
    const int J = mid_id<L>(t);  // = g + 16 i: thread i of sub-transform g
    const int g = J & 15, i = J >> 4;
    C2* x1 = sm + nat_id<L>(t) * IL;
#pragma unroll
    for (int m = 0; m < 16; ++m) x1[m * RS] = v[m];
    S::all();
    C2* own = sm + g * RS;
#pragma unroll
    for (int m = 0; m < 16; ++m) v[m] = own[i * IL + TG * m];
    fused_pass<L, 16, 16>(v, load_tw<L, 16, 16>(tab, J));
    S::in();
#pragma unroll
    for (int m = 0; m < 16; ++m) own[i * IL + TP * m] = v[m];
    S::in();
    if constexpr (L <= 4096) {
        constexpr int R3 = G::R3, B = 16 / R3;
#pragma unroll
        for (int b = 0; b < B; ++b)
#pragma unroll
            for (int r = 0; r < R3; ++r) v[b + r * B] = own[i * TP + G::TG * TP * b + r * IL];
        fused_pass<L, 16, 256>(v, load_tw<L, 16, 256>(tab, J));
    } else {
        const int k1 = i & 15, d = i >> 4;
        C2* q = own + k1 * TP;
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] = q[(2 * r + d) * IL];
        fused_pass<L, 16, 256>(v, load_tw<L, 16, 256>(tab, J));
#pragma unroll
        for (int m = 0; m < 16; ++m) q[(2 * m + d) * IL] = v[m];  // the slots this thread read
        S::in();
#pragma unroll
        for (int b = 0; b < 8; ++b)
#pragma unroll
            for (int r = 0; r < 2; ++r) v[b + 8 * r] = q[(4 * b + 2 * d + r) * IL];
        fused_pass<L, 16, 4096>(v, load_tw<L, 16, 4096>(tab, J));
    }
}

// `hook` runs once every thread of the block has read the line for the last
// time (a barrier then): from there on the line is free.
template <int L, class S, int IL = 1, class H = NoHook>
__device__ __forceinline__ void fft_second(C2 (&v)[16], C2* sm, const float2* __restrict__ tab, int t,
                                           const H& hook = H{}) {
    using G = Mirror<L>;
    constexpr int RS = G::RS * IL, TG = G::TG * IL, TP = TG + IL;  // in units of the interleaved line
    const int P = nat_id<L>(t);
    radix4_pass<L, 16, 1>(v, tab, t);
    S::in();
    if constexpr (L <= 4096) {
        constexpr int R3 = G::R3, NG = G::NG, B = 16 / R3;
        const int c = t >> 4, q = t & 15;  // group of 16 threads: mid ids equal to c modulo R3
        C2* grp = sm + c * RS;
        C2* w = grp + ((q % G::TG) + R3 * (q / G::TG)) * IL;
#pragma unroll
        for (int m = 0; m < 16; ++m) w[(m / R3) * R3 * RS + (m % R3) * 17 * IL] = v[m];
        S::in();
        const C2* x = grp + (q / R3) * R3 * RS + (q % R3) * 17 * IL;
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = x[((m / NG) + R3 * (m % NG)) * IL];
        fused_pass<L, 16, 16>(v, load_tw<L, 16, 16>(tab, P));
        S::in();
#pragma unroll
        for (int m = 0; m < 16; ++m) grp[q * IL + (m / G::TG) * R3 * RS + 16 * (m % G::TG) * IL] = v[m];
        S::all();
#pragma unroll
        for (int b = 0; b < B; ++b)
#pragma unroll
            for (int r = 0; r < R3; ++r) v[b + r * B] = sm[t * IL + (r + R3 * b) * RS];
        if constexpr (!H::none) {
            __syncthreads();
            hook();
        }
        fused_pass<L, 16, 256>(v, load_tw<L, 16, 256>(tab, P));
    } else {
        const int f = (t >> 4) & 1, k0 = t & 15, h = k0 + 16 * (t >> 5);
        C2* own = sm + (t >> 5) * RS;
#pragma unroll
        for (int m = 0; m < 16; ++m) own[(t & 31) * IL + TP * m] = v[m];
        S::in();
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] = own[k0 * TP + (2 * r + f) * IL];
        fused_pass<L, 16, 16>(v, load_tw<L, 16, 16>(tab, P));
        S::in();
#pragma unroll
        for (int m = 0; m < 16; ++m) own[(k0 + 256 * f + 16 * m) * IL] = v[m];
        S::all();
        C2* x = sm + f * RS + h * IL;
#pragma unroll
        for (int m = 0; m < 16; ++m) v[m] = x[2 * (m & 7) * RS + 256 * (m >> 3) * IL];
        fused_pass<L, 16, 256>(v, load_tw<L, 16, 256>(tab, P));
#pragma unroll
        for (int m = 0; m < 16; ++m) x[2 * (m & 7) * RS + 256 * (m >> 3) * IL] = v[m];  // the slots this thread read
        S::in();
        const C2* y = sm + 2 * f * RS + h * IL;
#pragma unroll
        for (int b = 0; b < 8; ++b)
#pragma unroll
            for (int r = 0; r < 2; ++r) v[b + 8 * r] = y[(4 * (b & 3) + r) * RS + 256 * (b >> 2) * IL];
        if constexpr (!H::none) {
            __syncthreads();
            hook();
        } else {
            S::in();  // the next use of the line may write slots the other half of the warp read
        }
        fused_pass<L, 16, 4096>(v, load_tw<L, 16, 4096>(tab, P));
    }
}

}  // namespace pr
}  // namespace nlse
