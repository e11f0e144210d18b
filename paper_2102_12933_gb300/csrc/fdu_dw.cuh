// Double-word arithmetic on FP32 pairs (device only).
//
// A double-word value x = h + l holds two FP32 numbers with |l| <= ulp(h)/2,
// about 48 significant bits.  The building blocks are the error-free
// transformations of Dekker and Knuth (2Sum, and the exact product error
// fma(a, b, -a*b)).  The kernels run on the lean forms at the end of this file;
// the normalised algorithms that these come from are in fdu_dw.cu, for the
// accuracy check.
//
// Every FP32 operation is an explicitly rounded intrinsic (__fadd_rn,
// __fmul_rn, __fmaf_rn): the compiler must not fuse a product into a later
// sum, which would break the error-free transformations.
#pragma once
#include <cuda_runtime.h>

namespace fdu {
namespace dwa {

// T = float: one double word; T = f2: two, one per lane of the packed FP32
// instructions (fadd2 / fmul2 / ffma2, one issue slot for two operations).
template <class T>
struct dwv {
    T h, l;
};
using dw = dwv<float>;

__device__ __forceinline__ dw dw_make(float h, float l = 0.0f) { return dw{h, l}; }

// s + t = a + b exactly, any order of magnitude
__device__ __forceinline__ dw two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float ap = __fsub_rn(s, b);
    const float bp = __fsub_rn(s, ap);
    return dw{s, __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp))};
}

// Compensated dot product (Ogita, Rump and Oishi, "Accurate sum and dot
// product", SIAM J. Sci. Comput. 26(6), 2005, algorithm Dot2, extended to
// double-word factors): s carries the running FP32 sum, c the sum of the
// exact errors of each product and sum plus the low-word cross terms; the
// result s + c has an absolute error of about u^2 times the sum of |terms|.
struct dot2 {
    float s, c;
};
__device__ __forceinline__ void dot2_add(dot2 &A, dw a, dw x) {
    const float p = __fmul_rn(a.h, x.h);
    const float e1 = __fmaf_rn(a.h, x.h, -p);
    const dw t = two_sum(A.s, p);
    A.s = t.h;
    A.c = __fadd_rn(A.c, __fadd_rn(__fadd_rn(e1, t.l), __fmaf_rn(a.h, x.l, __fmul_rn(a.l, x.h))));
}
__device__ __forceinline__ dw dot2_result(const dot2 &A) { return two_sum(A.s, A.c); }

// FP64 <-> double word by bit manipulation (GB300 runs float <-> double
// conversions on its FP64 pipe)
// double -> double word; magnitudes below 2^-126 flush to zero (the data
// stay far above); the high word keeps the top 24 bits (truncated), the low
// word the next 24 of the remaining 29 (relative error below 2^-47).  The
// pair is not renormalised (|l| < ulp(h) instead of ulp(h)/2): the
// operations that take it renormalise their results.  Magnitudes of 2^128 and
// above, infinities and NaN give an infinity or a NaN; BOUNDED leaves the test
// for them out, where the caller's values are known to be finite and smaller.
template <bool BOUNDED = false>
__device__ __forceinline__ dw d2dw(double d) {
    const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
    const int e = (int)((hi >> 20) & 0x7ffu);
    if (e <= 896) return dw_make(0.0f, 0.0f);
    const unsigned sgn = hi & 0x80000000u;
    const float h = __uint_as_float(sgn | ((unsigned)(BOUNDED ? e - 896 : min(e - 896, 255)) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
    const unsigned m = lo & 0x1fffffffu;  // value m 2^(e - 1075)
    const unsigned lb = __float_as_uint(__uint2float_rn(m));
    const int le = (int)((lb >> 23) & 0xffu) + (e - 1075);
    const float l = (m != 0u && le > 0) ? __uint_as_float(sgn | ((unsigned)le << 23) | (lb & 0x7fffffu)) : 0.0f;
    return dw_make(h, l);  // |l| < ulp(h): the truncated split, not renormalised
}
// float -> double, exact for finite normal floats (zero and subnormals -> 0)
__device__ __forceinline__ double f2d(float x) {
    const unsigned b = __float_as_uint(x);
    const unsigned e = (b >> 23) & 0xffu;
    if (e == 0u) return 0.0;
    return __hiloint2double((int)((b & 0x80000000u) | ((e + 896u) << 20) | ((b & 0x7fffffu) >> 3)), (int)(b << 29));
}
// a double word; a NaN where its high word is not finite
__device__ __forceinline__ double dw2d(dw x) {
    const double v = f2d(x.h) + f2d(x.l);
    return fabsf(x.h) < INFINITY ? v : __longlong_as_double(0x7ff8000000000000ll);
}

// ------------------------------------------------------------------ packed pairs, lean forms
// Two FP32 lanes in a 64-bit register pair, and the explicitly rounded
// operations on one lane (float) or two (f2).  GB300 issues a packed FP32
// instruction at half the scalar rate per instruction, that is at the same
// rate per element (measured: 3.64 FFMA against 1.88 FFMA2 warp instructions
// per clock and SM), so packing does not lift the FMA-pipe ceiling; it halves
// the issue slots and the instruction bytes, which is what the double-word
// kernels run out of first.  Negation and lane swaps of an operand cost
// nothing there (measured).
struct f2 {
    unsigned long long v;
};
using dw2 = dwv<f2>;
__device__ __forceinline__ f2 pk(float a, float b) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d.v) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ float lane0(f2 d) { return __uint_as_float((unsigned)d.v); }
__device__ __forceinline__ float lane1(f2 d) { return __uint_as_float((unsigned)(d.v >> 32)); }
__device__ __forceinline__ float fadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float ffma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float fneg(float a) { return -a; }
__device__ __forceinline__ f2 fadd(f2 a, f2 b) {
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ f2 fsub(f2 a, f2 b) {
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ f2 fmul(f2 a, f2 b) {
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d.v) : "l"(a.v), "l"(b.v));
    return d;
}
__device__ __forceinline__ f2 ffma(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return d;
}
__device__ __forceinline__ f2 fneg(f2 a) { return pk(-lane0(a), -lane1(a)); }
template <class T> __device__ __forceinline__ T splat(float a);
template <> __device__ __forceinline__ float splat<float>(float a) { return a; }
template <> __device__ __forceinline__ f2 splat<f2>(float a) { return pk(a, a); }
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ f2 rcp_approx(f2 x) { return pk(rcp_approx(lane0(x)), rcp_approx(lane1(x))); }
__device__ __forceinline__ f2 rsqrt_approx(f2 x) { return pk(rsqrt_approx(lane0(x)), rsqrt_approx(lane1(x))); }

__device__ __forceinline__ dw2 both(dw x) { return dw2{pk(x.h, x.h), pk(x.l, x.l)}; }       // (x, x)
__device__ __forceinline__ dw2 pair(dw a, dw b) { return dw2{pk(a.h, b.h), pk(a.l, b.l)}; }  // (a, b)
__device__ __forceinline__ dw2 swapped(dw2 x) {
    return dw2{pk(lane1(x.h), lane0(x.h)), pk(lane1(x.l), lane0(x.l))};
}
__device__ __forceinline__ dw first(dw2 x) { return dw{lane0(x.h), lane0(x.l)}; }
__device__ __forceinline__ dw second(dw2 x) { return dw{lane1(x.h), lane1(x.l)}; }

// The lean forms leave |l| up to a few ulp(h) (more after cancellation, at
// most about 2^-23 of the largest operand), which the products below take:
// every error stays near 2^-47 of the largest operand or product, the level
// of the sloppy sum, as long as one factor of each product is normalised (the
// product leaves out l l').  norm() restores |l| <= ulp(h)/2 for that, and
// where a sign or a comparison reads h.
template <class T>
__device__ __forceinline__ dwv<T> lneg(dwv<T> x) { return dwv<T>{fneg(x.h), fneg(x.l)}; }
template <class T>
__device__ __forceinline__ dwv<T> norm(dwv<T> x) {  // 3 operations; |h| >= |l|
    const T s = fadd(x.h, x.l);
    return dwv<T>{s, fsub(x.l, fsub(s, x.h))};
}
template <class T>
__device__ __forceinline__ dwv<T> ladd(dwv<T> x, dwv<T> y) {  // 8
    const T s = fadd(x.h, y.h);
    const T ap = fsub(s, y.h), bp = fsub(s, ap);
    const T e = fadd(fsub(x.h, ap), fsub(y.h, bp));
    return dwv<T>{s, fadd(e, fadd(x.l, y.l))};
}
template <class T>
__device__ __forceinline__ dwv<T> lsub(dwv<T> x, dwv<T> y) { return ladd(x, lneg(y)); }
template <class T>
__device__ __forceinline__ dwv<T> lmul(dwv<T> x, dwv<T> y) {  // 4
    const T p = fmul(x.h, y.h);
    return dwv<T>{p, ffma(x.l, y.h, ffma(x.h, y.l, ffma(x.h, y.h, fneg(p))))};
}
template <class T>
__device__ __forceinline__ dwv<T> lscale(dwv<T> x, float p2) {  // by a power of two: exact
    return dwv<T>{fmul(x.h, splat<T>(p2)), fmul(x.l, splat<T>(p2))};
}
// A + x y in 12 operations.  (Taking the product into the sum by one fused
// multiply-add and recovering the error as in 2Sum, 9 operations, is not
// error-free: with A near -x y the sum keeps bits of the product below ulp(A).)
template <class T>
__device__ __forceinline__ dwv<T> lfma(dwv<T> x, dwv<T> y, dwv<T> A) {
    const T p = fmul(x.h, y.h);
    const T s = fadd(A.h, p);
    const T ap = fsub(s, p), bp = fsub(s, ap);
    const T e = fadd(fsub(A.h, ap), fsub(p, bp));
    const T q = ffma(x.l, y.h, ffma(x.h, y.l, ffma(x.h, y.h, fneg(p))));
    return dwv<T>{s, fadd(e, fadd(A.l, q))};
}
// 1/x and 1/sqrt(x) from the hardware approximation (relative error below
// 2^-22) and one correction of second order in its residual; 1 - x.h r is one
// fused multiply-add, rounded at 2^-24 of the residual.
template <class T>
__device__ __forceinline__ dwv<T> lrecip(dwv<T> x) {  // 4 and the approximation
    const T r = rcp_approx(x.h);
    const T e = ffma(fneg(x.l), r, ffma(fneg(x.h), r, splat<T>(1.0f)));
    return dwv<T>{r, fmul(r, ffma(e, e, e))};
}
template <class T>
__device__ __forceinline__ dwv<T> lrsqrt(dwv<T> x) {  // 9 and the approximation
    const T y = rsqrt_approx(x.h);
    const T y2 = fmul(y, y), y2l = ffma(y, y, fneg(y2));
    const T e = fsub(ffma(fneg(x.h), y2, splat<T>(1.0f)), ffma(x.h, y2l, fmul(x.l, y2)));
    return dwv<T>{y, fmul(fmul(y, e), ffma(splat<T>(0.375f), e, splat<T>(0.5f)))};
}

}  // namespace dwa
}  // namespace fdu
