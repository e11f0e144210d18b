// Edge-flux VJP in double words (FP32 pairs, about 48 significant bits), which
// GB300 issues at 64 times its FP64 rate: the reverse sweep of the edge flux of
// fdu_dw_edge.cuh, in the same edge frame (momentum along the normal and the
// tangent) and with the left and right states in the two lanes of packed FP32
// instructions.  It differentiates the same function as the FP64 edge VJP
// (fdu_adjoint.cu) and takes the same branches (positivity fallback,
// entropy-fix band, sign of lambda).
//
// Precision 48 takes every edge here.  Precision 64 takes the edges whose
// derivative the double words hold to FP64's own accuracy and lists the others
// for the FP64 kernel (GUARD below); its FP64 kernel's one-step reciprocals are
// accurate to 2^-40, so the double words (2^-46) are the closer of the two:
// residual VJP of the 300^2 vortex against torch's autograd of the plain FP64
// residual 1.1e-13 in FP64, 1.6e-14 in double words.
//
// The nonlinear weights use the range-safe form of the forward kernel: per
// field the differences are scaled by lambda = 2^-K (max |difference| in
// [1/2, 1)) and beta' = lambda^2 (beta + eps), bounded below by 2^-100;
// omega = alpha / sum(alpha), alpha_k = C_k / beta'_k, and
//   d(out)/d(beta'_k) = -omega_k (v_k - out) / beta'_k,
//   d(beta'_k)/d(x)   = lambda (2 m0 x' + m1 y')  (x' = lambda x),
// zero where the bound holds beta' (a sub-stencil whose differences are
// below 2^-50 of the field's largest).
//
// What bounds it: the FMA pipe (53 % busy) behind instruction fetch (one stall
// per issue: the reverse is straight-line code) and the wait for dependent
// results at 10 to 12 warps per SM.  480k edges under ncu: 264 us, against 493
// us one operation to an instruction with normalised double words in x-y
// components, and 1092 us in FP64 (FP64 pipe 90 % busy).
#include <cuda_runtime.h>

#include <cstdint>

#include "fdu_adjoint.cuh"
#include "fdu_dw.cuh"
#include "fdu_dw_edge.cuh"
#include "fdu_dw_euler.cuh"
#include "fdu_internal.h"
#include "fdu_kernels.cuh"

namespace fdu {
namespace {

using namespace dwa;

constexpr int kVjpBlock = 64;
// per-thread 16-byte shared-memory slots, slot j of thread t at [j][t]
constexpr int kSlotBF = 0;   // fields' (b, f)
constexpr int kSlotAE = 4;   // fields' (a, e)
constexpr int kSlotC = 8;    // fields' c, two to a slot
constexpr int kSlotW = 10;   // per field (4 each): v1, v2, 1/B'_ad, 1/B'_bc; reverse: cotangents of ae, bf, c
constexpr int kSlotO = 26;   // per field: (dl, dr)
constexpr int kSlotB = 30;   // per field: cotangents of (dl, dr)
constexpr int kVjpSlots = 34;

template <class T>
__device__ __forceinline__ dwv<T> zero() { return dwv<T>{splat<T>(0.0f), splat<T>(0.0f)}; }
template <class T>
__device__ __forceinline__ void acc(dwv<T> &a, dwv<T> b) { a = ladd(a, b); }
template <class T>
__device__ __forceinline__ void fms(dwv<T> x, dwv<T> y, dwv<T> &A) { A = lfma(x, y, A); }
__device__ __forceinline__ dw sum2(dw2 x) { return ladd(first(x), second(x)); }
template <class T>
__device__ __forceinline__ vec4<T> norm4(const vec4<T> &v) { return vec4<T>{norm(v.x), norm(v.n), norm(v.t), norm(v.w)}; }
__device__ __forceinline__ vec4<f2> pair4(const vec4<float> &a, const vec4<float> &b) {
    return vec4<f2>{pair(a.x, b.x), pair(a.n, b.n), pair(a.t, b.t), pair(a.w, b.w)};
}
#define FDU_B(x) bcast(x, T{})

// State (rho, m_n, m_t, E) -> r = rho^-1/2, ir = 1/rho, p.
struct Prim2 {
    dw2 r, ir, p, ke2;  // ke2 = m_n^2 + m_t^2
};
struct Prim2Bar {
    dw2 r, ir, p;
};
__device__ __forceinline__ Prim2 prim2(const vec4<f2> &w, dw gm1) {
    Prim2 P;
    P.r = norm(lrsqrt(norm(w.x)));
    P.ir = norm(lmul(P.r, P.r));
    P.ke2 = norm(lfma(w.t, w.t, lmul(w.n, w.n)));
    P.p = norm(lmul(both(gm1), norm(lfma(lscale(P.ke2, -0.5f), P.ir, w.w))));
    return P;
}
__device__ __forceinline__ void prim2_vjp(const vec4<f2> &w, const Prim2 &P, const Prim2Bar &B, dw gm1, vec4<f2> &wb) {
    const dw2 pg = norm(lmul(B.p, both(gm1)));
    const dw2 irb = norm(lfma(lscale(pg, -0.5f), P.ke2, B.ir));
    const dw2 rb = norm(lfma(lscale(P.r, 2.0f), irb, B.r));
    fms(lscale(rb, -0.5f), norm(lmul(P.r, P.ir)), wb.x);  // d r / d rho = -r^3 / 2
    const dw2 g = norm(lmul(lneg(pg), P.ir));
    fms(g, w.n, wb.n);
    fms(g, w.t, wb.t);
    acc(wb.w, pg);
}
// Roe average of the two lanes, with 1 / (sum of sqrt(rho)) kept.
struct Roe2 {
    RoeN R;
    dw inv;
};
__device__ __forceinline__ Roe2 roe2(const vec4<f2> &w, const Prim2 &P, dw gm1) {
    Roe2 Q;
    Q.inv = norm(lrecip(norm(sum2(lmul(w.x, P.r)))));
    auto avg = [&](dw2 x) { return norm(lmul(norm(sum2(lmul(x, P.r))), Q.inv)); };
    Q.R = roe_n(avg(w.n), avg(w.t), avg(norm(ladd(w.w, P.p))), gm1);
    return Q;
}
// Cotangents of an average: q, t, H, c, hq2, and the raw sums sphi = sum phh_bar
// (c.x + c.w), spsi = sum psh_bar (c.x - c.w) of the projections, from which the
// parts through b1h = (gamma-1)/(2c^2) and ich = 1/(2c) follow.
template <class T>
struct RoeBar {
    dwv<T> q = zero<T>(), t = zero<T>(), H = zero<T>(), c = zero<T>(), hq2 = zero<T>(), sphi = zero<T>(),
           spsi = zero<T>();
};
__device__ __forceinline__ RoeBar<float> lanes(const RoeBar<f2> &B) {
    RoeBar<float> r;
    r.q = sum2(B.q);
    r.t = sum2(B.t);
    r.H = sum2(B.H);
    r.c = sum2(B.c);
    r.hq2 = sum2(B.hq2);
    r.sphi = sum2(B.sphi);
    r.spsi = sum2(B.spsi);
    return r;
}
__device__ __forceinline__ void add_bar(RoeBar<float> &a, const RoeBar<float> &b) {
    acc(a.q, b.q);
    acc(a.t, b.t);
    acc(a.H, b.H);
    acc(a.c, b.c);
    acc(a.hq2, b.hq2);
    acc(a.sphi, b.sphi);
    acc(a.spsi, b.spsi);
}
__device__ __forceinline__ void roe2_vjp(const vec4<f2> &w, const Prim2 &P, const Roe2 &Q, const RoeBar<float> &B,
                                         dw gm1, vec4<f2> &wb, Prim2Bar &Pb) {
    const RoeN &R = Q.R;
    const dw ic = lscale(R.ich, 2.0f);
    const dw icb = norm(lmul(R.c, norm(ladd(B.sphi, lscale(B.spsi, 0.5f)))));
    const dw c2b = norm(lmul(R.ich, norm(lfma(lneg(icb), norm(lmul(ic, ic)), B.c))));
    const dw c2g = norm(lmul(c2b, gm1));
    const dw Hb = norm(ladd(B.H, c2g)), hq2b = norm(lsub(B.hq2, c2g));
    const dw qb = norm(lfma(hq2b, R.q, B.q)), tb = norm(lfma(hq2b, R.t, B.t));
    const dw2 U = both(norm(lmul(qb, Q.inv))), V = both(norm(lmul(tb, Q.inv))), W = both(norm(lmul(Hb, Q.inv)));
    const dw2 sb = both(norm(lmul(lneg(lfma(Hb, R.H, lfma(tb, R.t, lmul(qb, R.q)))), Q.inv)));
    fms(sb, P.r, wb.x);
    fms(U, P.r, wb.n);
    fms(V, P.r, wb.t);
    const dw2 wr = lmul(W, P.r);
    acc(wb.w, wr);
    acc(Pb.p, wr);
    Pb.r = lfma(W, norm(ladd(w.w, P.p)), lfma(V, w.t, lfma(U, w.n, lfma(sb, w.x, Pb.r))));
}
// c = project_n(R, d): returns d's cotangent and adds R's, given the forward's
// acoustic fields c.x, c.w
template <class T>
__device__ __forceinline__ vec4<T> project_n_vjp(const RoeN &R, const vec4<T> &d, const dwv<T> &cx, const dwv<T> &cw,
                                                 const vec4<T> &cb, RoeBar<T> &B) {
    const dwv<T> q = FDU_B(R.q), t = FDU_B(R.t), hq2 = FDU_B(R.hq2);
    const dwv<T> phb = norm(lsub(ladd(cb.x, cb.w), lscale(cb.n, 2.0f))), psb = norm(lsub(cb.x, cb.w));
    fms(phb, ladd(cx, cw), B.sphi);
    fms(psb, lsub(cx, cw), B.spsi);
    const dwv<T> P = norm(lmul(phb, FDU_B(R.b1h))), U = norm(lmul(psb, FDU_B(R.ich)));
    const dwv<T> ctb = cb.t;
    fms(P, d.x, B.hq2);
    B.q = lfma(U, d.x, lfma(lneg(P), d.n, B.q));
    B.t = lfma(lneg(P), d.t, lfma(lneg(ctb), d.x, B.t));
    return vec4<T>{lfma(q, U, lfma(hq2, P, lfma(lneg(t), ctb, cb.n))), lfma(lneg(q), P, lneg(U)), lfma(lneg(t), P, ctb), P};
}
// out = unproject_n(R, c): c's cotangent and R's (added), from the cotangent ob of out
template <class T>
__device__ __forceinline__ vec4<T> unproject_n_vjp(const RoeN &R, const vec4<T> &c, const vec4<T> &ob, RoeBar<T> &B) {
    const dwv<T> q = FDU_B(R.q), t = FDU_B(R.t), cs = FDU_B(R.c);
    const dwv<T> ac = norm(ladd(c.x, c.w)), rho = norm(ladd(ac, c.n)), wx = norm(lsub(c.w, c.x)),
                 dd = norm(lmul(cs, wx));
    const dwv<T> rhob = lfma(t, ob.t, lfma(q, ob.n, ob.x)), ddb = norm(lfma(q, ob.w, ob.n));
    B.q = lfma(dd, ob.w, lfma(rho, ob.n, B.q));
    B.t = lfma(c.t, ob.w, lfma(rho, ob.t, B.t));
    fms(ac, ob.w, B.H);
    fms(c.n, ob.w, B.hq2);
    fms(wx, ddb, B.c);
    const dwv<T> acb = lfma(FDU_B(R.H), ob.w, rhob), cd = lmul(cs, ddb);
    return vec4<T>{norm(lsub(acb, cd)), norm(lfma(FDU_B(R.hq2), ob.w, rhob)), norm(lfma(t, ob.w, ob.t)),
                   norm(ladd(acb, cd))};
}
#undef FDU_B

// ---- NU-WENO5 of one field, both sides in the lanes (weno_pair_dw), keeping
// what the reverse needs
struct Scale {
    float lam;
    dw2 eps;
};
__device__ __forceinline__ Scale field_scale(dw2 ae, dw2 bf, dw2 bd, dw c, dw eps_m, int eps_e) {
    const float mx = fmaxf(fmaxf(fmaxf(fabsf(lane0(ae.h)), fabsf(lane1(ae.h))), fabsf(c.h)),
                           fmaxf(fmaxf(fabsf(lane0(bf.h)), fabsf(lane1(bf.h))), fabsf(lane1(bd.h))));
    const int be = bexp(mx), Ke = be == 0 ? 0 : be - 126;
    Scale s;
    s.lam = __uint_as_float((unsigned)(127 - Ke) << 23);
    const int e2 = min(eps_e - 2 * Ke, 100) + 127;
    s.eps = both(e2 >= 1 ? lscale(eps_m, __uint_as_float((unsigned)e2 << 23)) : dw_make(0.0f, 0.0f));
    return s;
}
__device__ __forceinline__ dw2 upper(dw c) { return dw2{pk(0.0f, c.h), pk(0.0f, c.l)}; }
__device__ __forceinline__ dw2 ldk(const float4 *kp, int64_t ne, int p) {
    const float4 q = __ldg(kp + (int64_t)p * ne);
    return dw2{pk(q.x, q.y), pk(q.z, q.w)};
}
__device__ __forceinline__ void weno_fwd(const float4 *kp, int64_t ne, dw2 ae, dw2 bf, dw c, dw eps_m, int eps_e,
                                         const Stage &S, int fi) {
    const dw2 c1 = upper(c), cc = both(c), bd = norm(ladd(bf, c1));
    const dw2 v1 = norm(lfma(ldk(kp, ne, 1), bf, lfma(ldk(kp, ne, 0), ae, c1)));
    const dw2 v2 = norm(lfma(ldk(kp, ne, 6), cc, lmul(ldk(kp, ne, 5), bd)));
    const Scale sc = field_scale(ae, bf, bd, c, eps_m, eps_e);
    const dw2 aes = lscale(ae, sc.lam), bfs = lscale(bf, sc.lam), bds = lscale(bd, sc.lam), cs = lscale(cc, sc.lam);
    const dw2 had = lfma(ldk(kp, ne, 3), bfs, lmul(ldk(kp, ne, 2), aes));
    dw2 Bad = norm(lfma(aes, had, lfma(ldk(kp, ne, 4), lmul(bfs, bfs), sc.eps)));
    const dw2 hbc = lfma(ldk(kp, ne, 8), cs, lmul(ldk(kp, ne, 7), bds));
    dw2 Bbc = norm(lfma(bds, hbc, lfma(ldk(kp, ne, 9), lmul(cs, cs), sc.eps)));
    Bad.h = at_least(Bad.h, 0x1p-100f);
    Bbc.h = at_least(Bbc.h, 0x1p-100f);
    const dw2 r1 = norm(lrecip(Bad)), r2 = norm(lrecip(Bbc));
    const dw2 l0 = lmul(ldk(kp, ne, 10), r1), l2 = lmul(ldk(kp, ne, 11), swapped(r2));
    const dw2 num = norm(lfma(l2, swapped(v2), lfma(r2, v2, lmul(l0, v1))));
    st_dw2(S, kSlotW + 4 * fi, v1);
    st_dw2(S, kSlotW + 4 * fi + 1, v2);
    st_dw2(S, kSlotW + 4 * fi + 2, r1);
    st_dw2(S, kSlotW + 4 * fi + 3, r2);
    st_dw2(S, kSlotO + fi, norm(lmul(num, norm(lrecip(norm(ladd(ladd(l0, r2), l2)))))));
}
// Reverse of one field from o = (cotangents of dl, dr): cotangents of ae, bf and
// c into the field's kSlotW slots.
__device__ __forceinline__ void weno_rev(const float4 *kp, int64_t ne, dw2 ae, dw2 bf, dw c, dw2 o, const Stage &S,
                                         int fi) {
    const dw2 v1 = ld_dw2(S, kSlotW + 4 * fi), v2 = ld_dw2(S, kSlotW + 4 * fi + 1);
    const dw2 r1 = ld_dw2(S, kSlotW + 4 * fi + 2), r2 = ld_dw2(S, kSlotW + 4 * fi + 3);
    const dw2 out = ld_dw2(S, kSlotO + fi);
    const dw2 l0 = lmul(ldk(kp, ne, 10), r1), l2 = lmul(ldk(kp, ne, 11), swapped(r2));
    const dw2 oi = norm(lmul(o, norm(lrecip(norm(ladd(ladd(l0, r2), l2))))));
    // o times the weights omega_0 (of v1), omega_1 (v2), omega_2 (v2 swapped)
    const dw2 o0 = norm(lmul(l0, oi)), o1 = norm(lmul(r2, oi)), o2 = norm(lmul(l2, oi));
    const dw2 v1b = o0, v2b = norm(ladd(o1, swapped(o2)));
    // cotangents of the scaled indicators: -omega_k (v_k - out) / B'_k over the sides that use them
    dw2 Bad = lneg(norm(lmul(norm(lmul(o0, norm(lsub(v1, out)))), r1)));
    const dw2 x2 = norm(lmul(o2, norm(lsub(swapped(v2), out))));
    dw2 Bbc = lneg(norm(lmul(norm(lfma(o1, norm(lsub(v2, out)), swapped(x2))), r2)));
    auto free_of_bound = [](dw2 B, dw2 r) {  // zero where beta' sits at its lower bound (1 / beta' = 2^100)
        const float m0 = lane0(r.h) < 0x1.fffffp99f ? 1.0f : 0.0f, m1 = lane1(r.h) < 0x1.fffffp99f ? 1.0f : 0.0f;
        const f2 m = pk(m0, m1);
        return dw2{fmul(B.h, m), fmul(B.l, m)};
    };
    Bad = free_of_bound(Bad, r1);
    Bbc = free_of_bound(Bbc, r2);
    const dw2 bd = norm(ladd(bf, upper(c)));
    const float lam = field_scale(ae, bf, bd, c, dw_make(0.0f), 0).lam;
    const dw2 aes = lscale(ae, lam), bfs = lscale(bf, lam), bds = lscale(bd, lam), cs = lscale(both(c), lam);
    const dw2 k2 = ldk(kp, ne, 2), k3 = ldk(kp, ne, 3), k7 = ldk(kp, ne, 7), k8 = ldk(kp, ne, 8);
    Bad = lscale(Bad, lam);
    Bbc = lscale(Bbc, lam);
    // beta = m0 x^2 + m1 x y + m2 y^2: slopes 2 m0 x + m1 y and m1 x + 2 m2 y
    const dw2 aeb = lfma(Bad, norm(lfma(k3, bfs, lmul(lscale(k2, 2.0f), aes))), lmul(ldk(kp, ne, 0), v1b));
    const dw2 bfb = lfma(Bad, norm(lfma(lscale(ldk(kp, ne, 4), 2.0f), bfs, lmul(k3, aes))), lmul(ldk(kp, ne, 1), v1b));
    const dw2 bdb = lfma(Bbc, norm(lfma(k8, cs, lmul(lscale(k7, 2.0f), bds))), lmul(ldk(kp, ne, 5), v2b));
    const dw2 ccb = lfma(Bbc, norm(lfma(lscale(ldk(kp, ne, 9), 2.0f), cs, lmul(k8, bds))), lmul(ldk(kp, ne, 6), v2b));
    // d = f + c; S_d's value counts c too
    const dw cb = ladd(ladd(sum2(ccb), second(bdb)), second(v1b));
    st_dw2(S, kSlotW + 4 * fi, norm(aeb));
    st_dw2(S, kSlotW + 4 * fi + 1, norm(ladd(bfb, bdb)));
    st_dw2(S, kSlotW + 4 * fi + 2, both(norm(cb)));
}

// float -> double times 2^k, exact for normal floats and results (zero and
// subnormals -> 0; results beyond the range -> 0 or infinity)
__device__ __forceinline__ double f2d_scaled(float x, int k) {
    const unsigned b = __float_as_uint(x), e = (b >> 23) & 0xffu;
    const int d = (int)e + 896 + k;
    if (e == 0u || d <= 0) return 0.0;
    if (d >= 2047) return __hiloint2double((int)((b & 0x80000000u) | 0x7ff00000u), 0);
    return __hiloint2double((int)((b & 0x80000000u) | ((unsigned)d << 20) | ((b & 0x7fffffu) >> 3)), (int)(b << 29));
}
__device__ __forceinline__ int dexp(double x) { return (int)(((unsigned)__double2hiint(x) >> 20) & 0x7ffu); }
// x times 2^-k (normal x and result; zero where it would not be normal)
__device__ __forceinline__ double scaled_down(double x, int k) {
    const int e = dexp(x) - k;
    if (dexp(x) == 0 || e <= 0) return 0.0;
    return __hiloint2double((__double2hiint(x) & (int)0x800fffff) | (e << 20), __double2loint(x));
}

// GUARD (precision 64): returns false for an edge that FP64 takes and writes: a
// state outside the forward kernel's density and energy window, differences that
// are not finite in FP32 (a NaN or huge momentum), an average whose c^2 is a small
// difference (edge_flux_dw_body), a cotangent that is not finite, a WENO epsilon so
// far below the state's squares that the derivative of the weights rests on the
// rounding of the differences (eps < 2^-76 max(rho, E)^2: noise of 2^-53 of the
// state, squared, would pass for an indicator; the fields are in units of density
// and momentum, |m|^2 < 2 rho E), outputs beyond FP32's range, or end states more
// than a factor of two apart in density or energy.  VJP against central
// differences in extended precision, FP64 / double words without the last line /
// with it, steps of 4, 16, 64 in density and pressure: 7.7e-14 / 1.4e-13 / 3.1e-14,
// 4.7e-14 / 2.6e-13 / 5.5e-14, 6.8e-14 / 3.9e-13 / 6.5e-14.  A line at 1.5 lists
// edges of smooth flow on coarse meshes (beta 5 vortex on 24^2 and 40^2: 71 and 75
// to 113 us) and gains nothing.
template <bool GUARD>
__device__ __forceinline__ bool edge_vjp_dw_body(const AdjEdgeArgs &A, const int64_t e, const Stage &S) {
    const double *__restrict__ w = A.w;
    const int64_t ne = A.ne;
    const float4 *kp = A.coefdw + e;
    const dw gm1 = dw_make(A.dw_gm1[0], A.dw_gm1[1]);
    int32_t s[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) s[i] = __ldg(A.sten + (int64_t)i * ne + e);
    const dw2 nn = ldk(kp, ne, kDwPairs - 1);
    const dw nx = first(nn), ny = second(nn);

    // the cotangent scaled by the power of two that brings its largest component to
    // [1, 2); as it is where one is not finite, which the split passes on
    d4v lam = ldd4(A.lam_r, e);
    const int big = max(max(dexp(lam.x), dexp(lam.y)), max(dexp(lam.z), dexp(lam.w)));
    const int kl = big == 2047 ? 0 : big - 1023;
    if (GUARD && (big == 2047 || (big == 0 && (lam.x != 0.0 || lam.y != 0.0 || lam.z != 0.0 || lam.w != 0.0)))) return false;
    lam = d4v{scaled_down(lam.x, kl), scaled_down(lam.y, kl), scaled_down(lam.z, kl), scaled_down(lam.w, kl)};

    // ---------------- forward
    const d4v L1d = ldd4(w, s[2]), R1d = ldd4(w, s[3]);
    if (GUARD) {
        // the high words of positive doubles order them, and 2^20 between two of them
        // is a factor of two
        const unsigned lo = (unsigned)(1023 - kWideExp) << 20, n = (unsigned)(2 * kWideExp) << 20;
        auto hi = [](double x) { return (unsigned)__double2hiint(x); };
        auto out = [&](const d4v &q) { return hi(q.x) - lo >= n || hi(q.w) - lo >= n; };
        auto jump = [&](double a, double b) { return hi(a) - hi(b) + (1u << 20) > 1u << 21; };
        bool bad = out(L1d) || out(R1d) || dexp(A.eps) < 2 * max(dexp(L1d.x), dexp(L1d.w)) - 1023 - 76;
        bad = bad || jump(L1d.x, R1d.x) || jump(L1d.w, R1d.w);
        bad = bad || out(ldd4(w, s[0])) || out(ldd4(w, s[1])) || out(ldd4(w, s[4])) || out(ldd4(w, s[5]));
        if (bad) return false;
    }
    auto diff = [](const d4v &p, const d4v &q) { return d2dw4(d4v{p.x - q.x, p.y - q.y, p.z - q.z, p.w - q.w}); };
    // differences of a stencil pair (left from L1, right from R1) in the edge's frame
    auto dpair = [&](int il, int ir) {
        const dw4 l = diff(ldd4(w, il), ldd4(w, s[2])), r = diff(ldd4(w, ir), ldd4(w, s[3]));
        vec4<f2> d;
        d.x = pair(l.x, r.x);
        d.w = pair(l.w, r.w);
        turn(nx, ny, pair(l.y, r.y), pair(l.z, r.z), d.n, d.t);
        return norm4(d);
    };
    auto dmid = [&]() {
        const dw4 m = diff(ldd4(w, s[3]), ldd4(w, s[2]));
        vec4<float> d;
        d.x = m.x;
        d.w = m.w;
        turn(nx, ny, m.y, m.z, d.n, d.t);
        return norm4(d);
    };
    vec4<f2> W1;  // (L1, R1)
    {
        const dw4 l = d2dw4(L1d), r = d2dw4(R1d);
        W1.x = norm(pair(l.x, r.x));
        W1.w = norm(pair(l.w, r.w));
        turn(nx, ny, pair(l.y, r.y), pair(l.z, r.z), W1.n, W1.t);
        W1.n = norm(W1.n);
        W1.t = norm(W1.t);
    }
    const Prim2 P1 = prim2(W1, gm1);
    const Roe2 C = roe2(W1, P1, gm1);
    if (GUARD && !(C.R.H.h - C.R.hq2.h >= 0.25f * C.R.H.h)) return false;
    {
        auto put = [&](const vec4<f2> &d, int slot) {
            const vec4<f2> c = project_n(C.R, d);
            st_dw2(S, slot, norm(c.x));
            st_dw2(S, slot + 1, norm(c.n));
            st_dw2(S, slot + 2, norm(c.t));
            st_dw2(S, slot + 3, norm(c.w));
        };
        put(dpair(s[1], s[4]), kSlotBF);
        put(dpair(s[0], s[5]), kSlotAE);
        const vec4<float> c = project_n(C.R, dmid());
        st_dw2(S, kSlotC, norm(pair(c.x, c.n)));
        st_dw2(S, kSlotC + 1, norm(pair(c.t, c.w)));
    }
    auto field_c = [&](int i) {
        const dw2 q = ld_dw2(S, kSlotC + (i >> 1));
        return (i & 1) ? second(q) : first(q);
    };
    {
        const dw eps_m = dw_make(A.dw_eps[0], A.dw_eps[1]);
#pragma unroll 1
        for (int i = 0; i < 4; ++i)
            weno_fwd(kp, ne, ld_dw2(S, kSlotAE + i), ld_dw2(S, kSlotBF + i), field_c(i), eps_m, A.dw_eps_e, S, i);
    }
    auto ld_out = [&]() {
        return vec4<f2>{ld_dw2(S, kSlotO), ld_dw2(S, kSlotO + 1), ld_dw2(S, kSlotO + 2), ld_dw2(S, kSlotO + 3)};
    };
    const vec4<f2> base{both(first(W1.x)), both(first(W1.n)), both(first(W1.t)), both(first(W1.w))};
    const vec4<f2> dd = norm4(unproject_n(C.R, ld_out()));
    vec4<f2> Wi{norm(ladd(base.x, dd.x)), norm(ladd(base.n, dd.n)), norm(ladd(base.t, dd.t)), norm(ladd(base.w, dd.w))};
    vec4<float> jump{lsub(second(dd.x), first(dd.x)), lsub(second(dd.n), first(dd.n)), lsub(second(dd.t), first(dd.t)),
                     lsub(second(dd.w), first(dd.w))};
    bool ok = lane0(Wi.x.h) > 0.0f && lane1(Wi.x.h) > 0.0f;
    Prim2 P = P1;
    if (ok) {
        P = prim2(Wi, gm1);
        ok = lane0(P.p.h) > 0.0f && lane1(P.p.h) > 0.0f;
    }
    if (!ok) {  // positivity fallback: the end states
        // not for differences beyond FP32's range, which leave a NaN in every state
        if (GUARD && !(lane0(dd.w.h) - lane0(dd.w.h) == 0.0f && lane1(dd.w.h) - lane1(dd.w.h) == 0.0f)) return false;
        Wi = W1;
        P = P1;
        jump = dmid();
    }
    jump = norm4(jump);
    const Roe2 Q = roe2(Wi, P, gm1);
    if (GUARD && !(Q.R.H.h - Q.R.hq2.h >= 0.25f * Q.R.H.h)) return false;
    const vec4<float> a = norm4(project_n(Q.R, jump));
    // nu = (l - |l|_fixed) / 2: min(l, 0), or -(l - delta)^2 / (4 delta) inside
    // Harten's band |l| < delta = 0.1 c, with d nu / d l and d nu / d delta =
    // (l^2 - delta^2) / (4 delta^2) (0 outside the band)
    const dw delta = norm(lmul(Q.R.c, dw_make(A.dw_tenth[0], A.dw_tenth[1])));
    const dw h4d = norm(lmul(Q.R.ich, dw_make(5.0f)));  // 1 / (4 delta)
    struct Wave {
        dw nu, gl, gd;
    };
    auto wave = [&](dw l) {
        const float ah = fabsf(l.h), al = l.h < 0.0f ? -l.l : l.l;
        const bool in = ah < delta.h || (ah == delta.h && al < delta.l), up = !(l.h < 0.0f);
        const dw sd = norm(lsub(l, delta)), sh = norm(lmul(sd, h4d));
        const dw nu = norm(lmul(lneg(sd), sh)), gl = lscale(sh, -2.0f),
                 gd = norm(lmul(lmul(norm(ladd(l, delta)), lscale(h4d, 4.0f)), sh));
        const dw z = dw_make(0.0f);
        return Wave{in ? nu : up ? z : l, in ? gl : up ? z : dw_make(1.0f), in ? gd : z};
    };
    const Wave wu = wave(Q.R.q), wm = wave(norm(lsub(Q.R.q, Q.R.c))), wp = wave(norm(ladd(Q.R.q, Q.R.c)));
    const vec4<float> sv{norm(lmul(wm.nu, a.x)), norm(lmul(wu.nu, a.n)), norm(lmul(wu.nu, a.t)), norm(lmul(wp.nu, a.w))};

    // ---------------- reverse
    vec4<float> ob;  // the cotangent in the edge's frame
    {
        const dw4 l = d2dw4(lam);
        ob.x = l.x;
        ob.w = l.w;
        turn(nx, ny, l.y, l.z, ob.n, ob.t);
        ob = norm4(ob);
    }
    vec4<f2> wb;  // cotangents of (w_L, w_R)
    Prim2Bar Pb{zero<f2>(), zero<f2>(), zero<f2>()};
    {
        // left physical flux (m_n, m_n q + p, m_t q, (E + p) q), q = m_n / rho
        const dw n = first(Wi.n), t = first(Wi.t), ir = first(P.ir), Ep = norm(ladd(first(Wi.w), first(P.p)));
        const dw q = norm(lmul(n, ir));
        const dw qb = norm(lfma(ob.w, Ep, lfma(ob.t, t, lmul(ob.n, n))));
        const dw z = dw_make(0.0f);
        wb.x = zero<f2>();
        wb.n = pair(lfma(qb, ir, lfma(ob.n, q, ob.x)), z);
        wb.t = pair(lmul(ob.t, q), z);
        wb.w = pair(lmul(ob.w, q), z);
        Pb.p = pair(lfma(ob.w, q, ob.n), z);
        Pb.ir = pair(lmul(qb, n), z);
    }
    {
        RoeBar<float> B;
        const vec4<float> svb = unproject_n_vjp(Q.R, sv, ob, B);
        const dw nmb = norm(lmul(a.x, svb.x)), nub = norm(lfma(a.t, svb.t, lmul(a.n, svb.n))), npb = norm(lmul(a.w, svb.w));
        const dw lub = lmul(nub, wu.gl), lmb = lmul(nmb, wm.gl), lpb = lmul(npb, wp.gl);
        B.q = ladd(B.q, ladd(lub, ladd(lmb, lpb)));
        const dw db = norm(lfma(npb, wp.gd, lfma(nmb, wm.gd, lmul(nub, wu.gd))));
        B.c = ladd(B.c, lfma(db, dw_make(A.dw_tenth[0], A.dw_tenth[1]), lsub(lpb, lmb)));
        const vec4<float> ab{norm(lmul(wm.nu, svb.x)), norm(lmul(wu.nu, svb.n)), norm(lmul(wu.nu, svb.t)),
                             norm(lmul(wp.nu, svb.w))};
        const vec4<float> jb = project_n_vjp(Q.R, jump, a.x, a.w, ab, B);
        acc(wb.x, pair(lneg(jb.x), jb.x));
        acc(wb.n, pair(lneg(jb.n), jb.n));
        acc(wb.t, pair(lneg(jb.t), jb.t));
        acc(wb.w, pair(lneg(jb.w), jb.w));
        roe2_vjp(Wi, P, Q, B, gm1, wb, Pb);
        prim2_vjp(Wi, P, Pb, gm1, wb);
    }
    wb = norm4(wb);
    double *G = A.G;  // [6][ne][4]
    float chk = 0.0f;  // 0 while every output is finite (else FP64 writes them all again)
    auto put = [&](int slot, dw x, dw n, dw t, dw v) {  // back to x-y components and to FP64, unscaled
        const dw2 m = norm(lfma(pair(lneg(ny), nx), both(t), lmul(pair(nx, ny), both(n))));
        auto to = [&](float h, float l) {
            const double v = f2d_scaled(h, kl) + f2d_scaled(l, kl);
            const bool odd = !GUARD && (__float_as_uint(h) & 0x7f800000u) == 0x7f800000u;
            return odd ? __hiloint2double(0x7ff80000, 0) : v;
        };
        if (GUARD) chk = fmaf(x.h, 0.0f, fmaf(lane0(m.h), 0.0f, fmaf(lane1(m.h), 0.0f, fmaf(v.h, 0.0f, chk))));
        double2 *q = reinterpret_cast<double2 *>(G + 4 * ((int64_t)slot * ne + e));
        q[0] = make_double2(to(x.h, x.l), to(lane0(m.h), lane0(m.l)));
        q[1] = make_double2(to(lane1(m.h), lane1(m.l)), to(v.h, v.l));
    };
    if (!ok) {
        const dw z = dw_make(0.0f);
        put(0, z, z, z, z);
        put(1, z, z, z, z);
        put(2, first(wb.x), first(wb.n), first(wb.t), first(wb.w));
        put(3, second(wb.x), second(wb.n), second(wb.t), second(wb.w));
        put(4, z, z, z, z);
        put(5, z, z, z, z);
        return !GUARD || chk == 0.0f;
    }
    // both interpolated states are L1 plus an increment
    const dw z = dw_make(0.0f);
    vec4<f2> g1{pair(sum2(wb.x), z), pair(sum2(wb.n), z), pair(sum2(wb.t), z), pair(sum2(wb.w), z)};  // of (L1, R1)
    RoeBar<f2> B2;
    const vec4<f2> ob2 = unproject_n_vjp(C.R, ld_out(), wb, B2);
    st_dw2(S, kSlotB, ob2.x);
    st_dw2(S, kSlotB + 1, ob2.n);
    st_dw2(S, kSlotB + 2, ob2.t);
    st_dw2(S, kSlotB + 3, ob2.w);
#pragma unroll 1
    for (int i = 0; i < 4; ++i)
        weno_rev(kp, ne, ld_dw2(S, kSlotAE + i), ld_dw2(S, kSlotBF + i), field_c(i), ld_dw2(S, kSlotB + i), S, i);
    auto cot = [&](int k) {  // cotangents of ae (k = 0), bf (1) or c (2) of the four fields
        return vec4<f2>{ld_dw2(S, kSlotW + k), ld_dw2(S, kSlotW + 4 + k), ld_dw2(S, kSlotW + 8 + k),
                        ld_dw2(S, kSlotW + 12 + k)};
    };
    // the two stencil pairs: cotangents of their states, and minus them of (L1, R1)
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        const int slot = k ? kSlotBF : kSlotAE;
        const vec4<f2> db = project_n_vjp(C.R, dpair(k ? s[1] : s[0], k ? s[4] : s[5]), ld_dw2(S, slot),
                                          ld_dw2(S, slot + 3), cot(k), B2);
        put(k, first(db.x), first(db.n), first(db.t), first(db.w));
        put(5 - k, second(db.x), second(db.n), second(db.t), second(db.w));
        g1 = vec4<f2>{lsub(g1.x, db.x), lsub(g1.n, db.n), lsub(g1.t, db.t), lsub(g1.w, db.w)};
    }
    {
        const vec4<f2> cc = cot(2);
        RoeBar<float> B;
        const vec4<float> db = project_n_vjp(C.R, dmid(), first(ld_dw2(S, kSlotC)), second(ld_dw2(S, kSlotC + 1)),
                                             vec4<float>{first(cc.x), first(cc.n), first(cc.t), first(cc.w)}, B);
        acc(g1.x, pair(lneg(db.x), db.x));
        acc(g1.n, pair(lneg(db.n), db.n));
        acc(g1.t, pair(lneg(db.t), db.t));
        acc(g1.w, pair(lneg(db.w), db.w));
        add_bar(B, lanes(B2));
        Prim2Bar Pc{zero<f2>(), zero<f2>(), zero<f2>()};
        roe2_vjp(W1, P1, C, B, gm1, g1, Pc);
        prim2_vjp(W1, P1, Pc, gm1, g1);
    }
    put(2, first(g1.x), first(g1.n), first(g1.t), first(g1.w));
    put(3, second(g1.x), second(g1.n), second(g1.t), second(g1.w));
    return !GUARD || chk == 0.0f;
}

// At most 200 registers, 5 blocks (10 warps) per SM: 0.270 ms for the residual
// VJP of 90,000 vertices (transposes included), 0.274 with 6 and 0.273 with 4.
template <bool GUARD>
__global__ void __launch_bounds__(kVjpBlock, 5) edge_flux_vjp_dw_kernel(const __grid_constant__ AdjEdgeArgs A) {
    __shared__ float4 stage[kVjpSlots * kVjpBlock];
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= A.ne) return;
    if (!edge_vjp_dw_body<GUARD>(A, e, Stage{stage + threadIdx.x, kVjpBlock})) A.list[atomicAdd(A.nlist, 1)] = (int32_t)e;
}

}  // namespace

void launch_edge_flux_vjp_dw(const AdjEdgeArgs &a, cudaStream_t s) {
    if (a.ne <= 0) return;
    const unsigned g = (unsigned)((a.ne + kVjpBlock - 1) / kVjpBlock);
    if (a.prec == 48) edge_flux_vjp_dw_kernel<false><<<g, kVjpBlock, 0, s>>>(a);
    else edge_flux_vjp_dw_kernel<true><<<g, kVjpBlock, 0, s>>>(a);
}

}  // namespace fdu
