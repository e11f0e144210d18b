// The precision-48 edge flux (device only): NU-WENO5 of one field in
// double words and the edge-flux body, shared by the standalone kernel
// (fdu_dw.cu) and the batched persistent stage (fdu_kernels.cu).  See
// fdu_dw.cu for the arithmetic's design.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "fdu_dw.cuh"
#include "fdu_dw_euler.cuh"
#include "fdu_internal.h"
#include "fdu_kernels.cuh"

namespace fdu {
namespace dwa {

// ---- NU-WENO5 increments of one field, both sides at once: lane 0 is the
// left state, lane 1 the right (mirrored) one.  The right side's sub-stencils
// are the left side's seen from R1, so every step of the two sides is the same
// operation on paired operands: S_a with S_d, S_b with S_c (the sub-stencils
// of weno_pair64_l1; right increments from L1).
//   ae = (a, e) = (L3-L1, R3-R1), bf = (b, f) = (L2-L1, R2-R1), c = R1-L1,
//   d = f + c = R2-L1 (characteristic components of one field)
// K: the edge's paired coefficients (kDwPairs, fdu_internal.h).
__device__ __forceinline__ int bexp(float x) { return (int)((__float_as_uint(x) >> 23) & 0xffu); }
__device__ __forceinline__ f2 at_least(f2 x, float m) { return pk(fmaxf(lane0(x), m), fmaxf(lane1(x), m)); }

__device__ __forceinline__ dw2 weno_pair_dw(const dw2 *K, dw2 ae, dw2 bf, dw c, dw eps_m, int eps_e) {
    const dw2 c1{pk(0.0f, c.h), pk(0.0f, c.l)}, cc = both(c);
    const dw2 bd = norm(ladd(bf, c1));                                  // (b, d)
    const dw2 v1 = norm(lfma(K[1], bf, lfma(K[0], ae, c1)));            // (v_a, v_d + c): S_d's value from L1
    const dw2 v2 = norm(lfma(K[6], cc, lmul(K[5], bd)));                // (v_b, v_c)
    // common power-of-two scale of the six differences: max |.| in [1/2, 1)
    const float mx = fmaxf(fmaxf(fmaxf(fabsf(lane0(ae.h)), fabsf(lane1(ae.h))), fabsf(c.h)),
                           fmaxf(fmaxf(fabsf(lane0(bf.h)), fabsf(lane1(bf.h))), fabsf(lane1(bd.h))));
    const int be = bexp(mx);
    const int Ke = be == 0 ? 0 : be - 126;                           // mx in [2^(Ke-1), 2^Ke)
    const float lam = __uint_as_float((unsigned)(127 - Ke) << 23);  // 2^-Ke (Ke in [-125, 128])
    const dw2 aes = lscale(ae, lam), bfs = lscale(bf, lam), bds = lscale(bd, lam);
    const dw cs = lscale(c, lam);
    // eps 2^(-2Ke) = eps_m 2^(eps_e - 2Ke) (zero below the float range)
    const int e2 = min(eps_e - 2 * Ke, 100) + 127;  // beyond 2^100 the weights are the linear ones anyway
    const dw2 eps = both(e2 >= 1 ? lscale(eps_m, __uint_as_float((unsigned)e2 << 23)) : dw_make(0.0f, 0.0f));
    // beta + eps = x (m0 x + m1 y) + m2 y^2 + eps, held above 2^-100
    const dw2 had = lfma(K[3], bfs, lmul(K[2], aes));
    dw2 Bad = norm(lfma(aes, had, lfma(K[4], lmul(bfs, bfs), eps)));
    const dw2 hbc = lfma(K[8], both(cs), lmul(K[7], bds));
    dw2 Bbc = norm(lfma(bds, hbc, lfma(K[9], both(lmul(cs, cs)), eps)));
    Bad.h = at_least(Bad.h, 0x1p-100f);
    Bbc.h = at_least(Bbc.h, 0x1p-100f);
    const dw2 r1 = lrecip(Bad), r2 = lrecip(Bbc), r3 = swapped(r2);
    // alpha_k = C_k / (beta_k + eps); the block stores C_0/C_1, C_2/C_1 (C_1 -> 1)
    const dw2 l0 = lmul(K[10], r1), l2 = lmul(K[11], r3);
    const dw2 num = norm(lfma(l2, swapped(v2), lfma(r2, v2, lmul(l0, v1))));
    return norm(lmul(num, norm(lrecip(norm(ladd(ladd(l0, r2), l2))))));
}

// ---- the edge flux, in the edge's frame: a state's momentum is kept as its
// components along the normal n and the tangent t = (-n_y, n_x), which the
// flux along the edge does not mix, and the result is turned back at the end.
// Against x-y components this drops the two direction products from every
// projection, back-projection, Roe average and flux.
// A 4-vector (rho, m_n, m_t, rho E) or (fields q_n - c, entropy, shear, q_n + c).
template <class T>
struct vec4 {
    dwv<T> x, n, t, w;
};
struct RoeN {  // Roe average along the edge: q_n, q_t, H, c, (q_n^2 + q_t^2)/2, (gamma-1)/(2c^2), 1/(2c)
    dw q, t, H, c, hq2, b1h, ich;
};
__device__ __forceinline__ RoeN roe_n(dw q, dw t, dw H, dw gm1) {
    RoeN R;
    R.q = q;
    R.t = t;
    R.H = norm(H);
    R.hq2 = norm(lscale(lfma(t, t, lmul(q, q)), 0.5f));
    const dw c2 = norm(lmul(gm1, norm(lsub(R.H, R.hq2))));
    const dw ic = norm(lrsqrt(c2));
    R.c = norm(lmul(c2, ic));
    R.b1h = norm(lscale(lmul(gm1, lmul(ic, ic)), 0.5f));
    R.ich = lscale(ic, 0.5f);
    return R;
}
__device__ __forceinline__ dw bcast(dw x, float) { return x; }
__device__ __forceinline__ dw2 bcast(dw x, f2) { return both(x); }
#define FDU_B(x) bcast(x, T{})
template <class T>
__device__ __forceinline__ vec4<T> project_n(const RoeN &R, const vec4<T> &d) {
    const dwv<T> q = FDU_B(R.q), t = FDU_B(R.t);
    const dwv<T> phh = lmul(FDU_B(R.b1h), lfma(lneg(t), d.t, lfma(lneg(q), d.n, lfma(FDU_B(R.hq2), d.x, d.w))));
    const dwv<T> psh = lmul(FDU_B(R.ich), lfma(q, d.x, lneg(d.n)));
    return vec4<T>{ladd(phh, psh), lsub(d.x, lscale(phh, 2.0f)), lfma(lneg(t), d.x, d.t), lsub(phh, psh)};
}
template <class T>
__device__ __forceinline__ vec4<T> unproject_n(const RoeN &R, const vec4<T> &c) {
    const dwv<T> q = FDU_B(R.q), t = FDU_B(R.t);
    const dwv<T> ac = ladd(c.x, c.w), rho = ladd(ac, c.n), dd = lmul(FDU_B(R.c), lsub(c.w, c.x));
    return vec4<T>{rho, lfma(q, rho, dd), lfma(t, rho, c.t),
                   lfma(t, c.t, lfma(q, dd, lfma(FDU_B(R.hq2), c.n, lmul(FDU_B(R.H), ac))))};
}
// (x, y) momentum components to (n, t) ones
template <class T>
__device__ __forceinline__ void turn(dw nx, dw ny, dwv<T> mx, dwv<T> my, dwv<T> &n, dwv<T> &t) {
    const dwv<T> a = FDU_B(nx), b = FDU_B(ny);
    n = lfma(b, my, lmul(a, mx));
    t = lfma(lneg(b), mx, lmul(a, my));
}

// Per-thread staging in shared memory, 16-byte slot j of thread t at [j][t]:
// the four fields' (b, f), (a, e) and, two to a slot, c; the increments (dl,
// dr) take the (b, f) slots.  The fields run as a loop over the staged values:
// unrolled by two or four the kernel is slower (0.1167 and 0.137 ms against
// 0.1146 ms at 250k vertices), its code then overflows the instruction caches.
constexpr int kDwSlots = 10;
// slot j of a thread at S[j * stride] (stride = the threads of the block)
struct Stage {
    float4 *S;
    int stride;
};
__device__ __forceinline__ void st_dw2(const Stage &T, int j, dw2 v) {
    T.S[j * T.stride] = make_float4(lane0(v.h), lane1(v.h), lane0(v.l), lane1(v.l));
}
__device__ __forceinline__ dw2 ld_dw2(const Stage &T, int j) {
    const float4 q = T.S[j * T.stride];
    return dw2{pk(q.x, q.y), pk(q.z, q.w)};
}

// The slots that the first two stages write, cleared in the first stage, and the
// slot of the step's result, cleared in the third stage just before that stage
// writes it: a caller may stop after the second stage and keep the start state.
__device__ __forceinline__ void clear_wide(const EdgeArgs &A, int64_t e) {
    if (!A.wide || e > A.n_comp) return;
    int *f = A.wide + kWideSlots * e;  // e: all meshes of a batch, or the one mesh (0), and each of a batch's
    if (A.wide_in == 0) f[1] = f[2] = 0;
    if (A.wide_in == 2) f[0] = 0;
}

// Writes the increment of edge e and returns true.  With GUARD (precision 64)
// the states are in the window (outside_window: no NaN, nothing beyond FP32's
// range), and it returns false, writing nothing, where the double words would lose
// more than FP64 does, and the caller takes the edge in FP64:
//  - an average whose c^2 is a small difference, (H - q^2/2) < H/4 (Mach numbers
//    above sqrt(6 / (gamma - 1)), 3.9 for gamma = 1.4), costs the double words
//    log2(H / (H - q^2/2)) of their 48 bits (measured on the flux itself against
//    extended precision: at amplitude 0.3 over 48 vertices 3e-16 at Mach 1, 7e-16
//    at 3, 7e-15 at 10);
//  - a state thinner than L1/64 formed from L1 costs log2 of that ratio.  Residual
//    against extended precision, FP64 / double words without this / with it, flow
//    across density steps of 64, 256, 1024, 4096: 2.1e-14 / 3.7e-15 / 5e-15, 2.4e-14
//    / 1.6e-14 / 1.2e-14, 2.6e-14 / 1.5e-13 / 1.7e-14, 4.5e-14 / 1.4e-12 / 4e-14.
template <bool GUARD>
__device__ __forceinline__ bool edge_flux_dw_body(const EdgeArgs &A, const int64_t e, const Stage &S) {
    const double *__restrict__ w = static_cast<const double *>(A.w);
    const int64_t ne = A.ne;
    const dw gm1 = dw_make(A.dw_gm1[0], A.dw_gm1[1]);
    int32_t s[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) s[i] = __ldg(A.sten + (int64_t)i * ne + e);
    const float4 nq = __ldg(A.coefdw + (int64_t)(kDwPairs - 1) * ne + e);
    const dw nx = dw_make(nq.x, nq.z), ny = dw_make(nq.y, nq.w);

    // Roe average of the end states from their records (the two summed in FP64)
    RoeN C;
    {
        const d4v qa = ldd4(A.Q, s[2]), qb = ldd4(A.Q, s[3]);
        const dw4 q = d2dw4<GUARD>(d4v{qa.x + qb.x, qa.y + qb.y, qa.z + qb.z, qa.w + qb.w});
        const dw inv = norm(lrecip(q.x));
        dw mn, mt;
        turn(nx, ny, q.y, q.z, mn, mt);
        C = roe_n(norm(lmul(mn, inv)), norm(lmul(mt, inv)), lmul(q.w, inv), gm1);
        if (GUARD && !(C.H.h - C.hq2.h >= 0.25f * C.H.h)) return false;
    }
    vec4<float> b;  // L1
    {
        // FP64 differences, then double words in the edge's frame and their
        // characteristic components: (L2-L1, R2-R1) and (L3-L1, R3-R1) paired, R1-L1
        const d4v L1 = ldd4(w, s[2]), R1 = ldd4(w, s[3]);
        auto diff = [](const d4v &p, const d4v &q) { return d2dw4<GUARD>(d4v{p.x - q.x, p.y - q.y, p.z - q.z, p.w - q.w}); };
        auto two = [&](int il, int ir, int slot) {
            const dw4 l = diff(ldd4(w, il), L1), r = diff(ldd4(w, ir), R1);
            vec4<f2> d;
            d.x = pair(l.x, r.x);
            d.w = pair(l.w, r.w);
            turn(nx, ny, pair(l.y, r.y), pair(l.z, r.z), d.n, d.t);
            const vec4<f2> c = project_n(C, d);
            st_dw2(S, slot, norm(c.x));
            st_dw2(S, slot + 1, norm(c.n));
            st_dw2(S, slot + 2, norm(c.t));
            st_dw2(S, slot + 3, norm(c.w));
        };
        two(s[1], s[4], 0);
        two(s[0], s[5], 4);
        const dw4 m = diff(R1, L1), l = d2dw4<GUARD>(L1);
        vec4<float> d;
        d.x = m.x;
        d.w = m.w;
        turn(nx, ny, m.y, m.z, d.n, d.t);
        const vec4<float> c = project_n(C, d);
        st_dw2(S, 8, norm(pair(c.x, c.n)));
        st_dw2(S, 9, norm(pair(c.t, c.w)));
        b.x = l.x;
        b.w = l.w;
        turn(nx, ny, l.y, l.z, b.n, b.t);
        b.n = norm(b.n);
        b.t = norm(b.t);
    }
    {
        dw2 K[kDwPairs - 1];
#pragma unroll
        for (int i = 0; i < kDwPairs - 1; ++i) {
            const float4 q = __ldg(A.coefdw + (int64_t)i * ne + e);
            K[i] = dw2{pk(q.x, q.y), pk(q.z, q.w)};
        }
        const dw eps_m = dw_make(A.dw_eps[0], A.dw_eps[1]);
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {
            const dw2 cq = ld_dw2(S, 8 + (i >> 1));
            st_dw2(S, i, weno_pair_dw(K, ld_dw2(S, 4 + i), ld_dw2(S, i), (i & 1) ? second(cq) : first(cq), eps_m,
                                      A.dw_eps_e));
        }
    }

    // primitives of L1
    const dw ib = norm(lrecip(b.x));
    const dw qnb = norm(lmul(b.n, ib)), qtb = norm(lmul(b.t, ib));
    const dw mu = lfma(b.t, qtb, lmul(b.n, qnb));  // |m|^2 / rho
    const dw pb = norm(lmul(gm1, lsub(b.w, lscale(mu, 0.5f))));

    // increments of both interpolated states (left, right) from L1
    vec4<f2> dd = unproject_n(C, vec4<f2>{ld_dw2(S, 0), ld_dw2(S, 1), ld_dw2(S, 2), ld_dw2(S, 3)});
    dd = vec4<f2>{norm(dd.x), norm(dd.n), norm(dd.t), norm(dd.w)};
    // the states from their increments: rho', 1/sqrt(rho'), the normal velocity
    // and pressure increments
    struct Sides {
        dw2 rho, r, dq, dp, p;
    } P;
    auto sides = [&]() {
        P.rho = norm(ladd(both(b.x), dd.x));
        if (!(lane0(P.rho.h) > 0.0f && lane1(P.rho.h) > 0.0f)) return false;
        P.r = norm(lrsqrt(P.rho));
        const dw2 ir = norm(lmul(P.r, P.r));
        P.dq = norm(lmul(lfma(both(lneg(qnb)), dd.x, dd.n), ir));
        // K' - K = ((2m + dm).dm - (|m|^2/rho) drho) / (2 rho')
        const dw2 k2 = lfma(both(lneg(mu)), dd.x,
                            lfma(ladd(both(lscale(b.t, 2.0f)), dd.t), dd.t,
                                 lmul(ladd(both(lscale(b.n, 2.0f)), dd.n), dd.n)));
        P.dp = lmul(both(gm1), lfma(lscale(k2, -0.5f), ir, dd.w));
        P.p = norm(ladd(both(pb), P.dp));
        return lane0(P.p.h) > 0.0f && lane1(P.p.h) > 0.0f;
    };
    bool fell_back = false;
    if (!sides()) {  // positivity fallback: first-order end states
        const d4v L1 = ldd4(w, s[2]), R1 = ldd4(w, s[3]);
        const dw4 m = d2dw4<GUARD>(d4v{R1.x - L1.x, R1.y - L1.y, R1.z - L1.z, R1.w - L1.w});
        const dw z = dw_make(0.0f);
        dw n, t;
        turn(nx, ny, m.y, m.z, n, t);
        dd = vec4<f2>{pair(z, m.x), pair(z, n), pair(z, t), pair(z, m.w)};
        sides();
        fell_back = true;
    }

    if (GUARD && !(fminf(lane0(P.rho.h), lane1(P.rho.h)) >= 0.015625f * b.x.h)) return false;

    // flux increment F_n(w_L) - F_n(L1)
    const vec4<float> il{first(dd.x), first(dd.n), first(dd.t), first(dd.w)};
    const dw dql = first(P.dq), dpl = first(P.dp);
    const dw qnl = norm(ladd(qnb, dql));
    vec4<float> out;
    out.x = il.n;
    out.n = lfma(b.n, dql, lfma(il.n, qnl, dpl));
    out.t = lfma(b.t, dql, lmul(il.t, qnl));
    out.w = lfma(ladd(b.w, pb), dql, lmul(ladd(il.w, dpl), qnl));

    // Roe dissipation at the Roe average of (w_L, w_R)
    {
        const dw2 sr = lmul(P.rho, P.r);
        const dw inv = norm(lrecip(ladd(first(sr), second(sr))));
        auto avg = [&](dw2 x) {
            const dw2 y = lmul(x, P.r);
            return lmul(ladd(first(y), second(y)), inv);
        };
        const RoeN Q = roe_n(norm(avg(ladd(both(b.n), dd.n))), norm(avg(ladd(both(b.t), dd.t))),
                             avg(ladd(ladd(both(b.w), dd.w), P.p)), gm1);
        if (GUARD && !(Q.H.h - Q.hq2.h >= 0.25f * Q.H.h)) return false;
        const vec4<float> a = project_n(Q, vec4<float>{lsub(second(dd.x), il.x), lsub(second(dd.n), il.n),
                                                       lsub(second(dd.t), il.t), lsub(second(dd.w), il.w)});
        // (l - |l|_fixed) / 2: min(l, 0), or -(l - delta)^2 / (4 delta) inside Harten's band |l| < delta = 0.1 c
        const dw delta = norm(lmul(Q.c, dw_make(A.dw_tenth[0], A.dw_tenth[1])));
        const dw h4d = norm(lmul(Q.ich, dw_make(5.0f)));  // 1 / (4 delta)
        auto fixed = [&](float lh, float ll, float fh, float fl) {
            const float ah = fabsf(lh), al = lh < 0.0f ? -ll : ll;
            const bool in = ah < delta.h || (ah == delta.h && al < delta.l);
            const bool up = !(lh < 0.0f);
            return dw_make(in ? -fh : up ? 0.0f : lh, in ? -fl : up ? 0.0f : ll);
        };
        const dw2 lmp = norm(ladd(both(Q.q), pair(lneg(Q.c), Q.c)));  // q_n - c, q_n + c
        const dw2 smp = norm(lsub(lmp, both(delta)));
        const dw2 fmp = norm(lmul(lmul(smp, smp), both(h4d)));
        const dw su = norm(lsub(Q.q, delta)), fu = norm(lmul(lmul(su, su), h4d));
        const dw nm = fixed(lane0(lmp.h), lane0(lmp.l), lane0(fmp.h), lane0(fmp.l));
        const dw np = fixed(lane1(lmp.h), lane1(lmp.l), lane1(fmp.h), lane1(fmp.l));
        const dw nu = fixed(Q.q.h, Q.q.l, fu.h, fu.l);
        const vec4<float> D = unproject_n(Q, vec4<float>{lmul(nm, a.x), lmul(nu, a.n), lmul(nu, a.t), lmul(np, a.w)});
        out.x = ladd(out.x, D.x);
        out.n = ladd(out.n, D.n);
        out.t = ladd(out.t, D.t);
        out.w = ladd(out.w, D.w);
    }

    // the increment r - F_n(L1), back in x-y components; the divergence adds
    // F_n(L1) through its folded vertex weights
    const dw2 m = norm(lfma(pair(lneg(ny), nx), both(out.t), lmul(pair(nx, ny), both(out.n))));
    const dw2 xw = norm(pair(out.x, out.w));
    float4 *r = static_cast<float4 *>(A.r);
    r[2 * e] = make_float4(lane0(xw.h), lane0(xw.l), lane0(m.h), lane0(m.l));
    r[2 * e + 1] = make_float4(lane1(m.h), lane1(m.l), lane1(xw.h), lane1(xw.l));
    if (fell_back) atomicAdd(A.fallback, 1ull);
    return true;
}
#undef FDU_B

}  // namespace dwa
}  // namespace fdu
