// sm_103a kernels of the unstructured-mesh FDM residual and SSP-RK3 stage.
//
//   edge flux  : per edge, gather the six states of its 1D curvilinear
//                stencil, project differences on the characteristic
//                fields of the Roe average of the edge's end states,
//                interpolate each field to the edge midpoint with
//                non-uniform WENO5 from both sides (Appendix), back-project
//                and evaluate a Roe flux along the edge (Section 2.3.1).
//   divergence : per vertex, a1 + b2 of the least-squares fit, i.e. the
//                weighted sum of vertex fluxes f_j, g_j and edge fluxes r_k
//                (Section 2.2.1), SELL-32 layout (a warp reads 32
//                consecutive ids / weights per entry); optionally fused
//                with the SSP-RK3 stage combination and the vertex fluxes
//                of the new state.
//
// Everything is gather-bound or scalar-ALU-bound: there is no dense
// contraction, so no tensor-core path.
#include <cuda_runtime.h>

#include <cstdint>

#include "fdu_internal.h"
#include "fdu_kernels.cuh"
#include "fdu_device.cuh"
#include "fdu_dw.cuh"
#include "fdu_dw_edge.cuh"

namespace fdu {
namespace {

using namespace dev;

// ------------------------------------------------------------------ FP64 edge flux
__device__ __forceinline__ dbl4 edge_flux_f64_value(const EdgeArgs &A, const int64_t e) {
    const double *__restrict__ w = static_cast<const double *>(A.w);
    const double *__restrict__ coef = static_cast<const double *>(A.coef);
    const double gm1 = A.gm1, hgm1 = A.hgm1;
    const int64_t ne = A.ne;
    int32_t s[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) s[i] = __ldg(A.sten + (int64_t)i * ne + e);
    const dbl4 L1 = ld4v(w, s[2]), R1 = ld4v(w, s[3]);
    const double nx = __ldg(coef + (int64_t)kCoefN * ne + e);
    const double ny = __ldg(coef + (int64_t)(kCoefN + 1) * ne + e);

    // characteristic decomposition at the Roe average of the end states
    // (per-vertex Roe records when the stage kernel provided them)
    const Roe64 C = A.Q ? roe64_from_records(ld4v(A.Q, s[2]), ld4v(A.Q, s[3]), nx, ny, gm1, hgm1)
                        : roe64(L1, prim64(L1, gm1), R1, prim64(R1, gm1), nx, ny, gm1, hgm1);
    const dbl4 cM = project64(C, sub4(R1, L1));               // R1 - L1
    const dbl4 cL2 = project64(C, sub4(ld4v(w, s[1]), L1));    // L2 - L1
    const dbl4 cL3 = project64(C, sub4(ld4v(w, s[0]), L1));    // L3 - L1
    const dbl4 cR2 = project64(C, sub4(ld4v(w, s[4]), R1));    // R2 - R1
    const dbl4 cR3 = project64(C, sub4(ld4v(w, s[5]), R1));    // R3 - R1

    double k[kCoefN];
#pragma unroll
    for (int i = 0; i < kCoefN; ++i) k[i] = __ldg(coef + (int64_t)i * ne + e);
    const dbl4 cR2L = add4(cR2, cM);  // R2 - L1
    dbl4 dl, dr;
    weno_pair64_l1(k, cL3.x, cL2.x, cM.x, cR2L.x, cR3.x, cR2.x, A.eps, dl.x, dr.x);
    weno_pair64_l1(k, cL3.y, cL2.y, cM.y, cR2L.y, cR3.y, cR2.y, A.eps, dl.y, dr.y);
    weno_pair64_l1(k, cL3.z, cL2.z, cM.z, cR2L.z, cR3.z, cR2.z, A.eps, dl.z, dr.z);
    weno_pair64_l1(k, cL3.w, cL2.w, cM.w, cR2L.w, cR3.w, cR2.w, A.eps, dl.w, dr.w);

    // both interpolated states from L1 (R (R1 - L1)_char = R1 - L1)
    dbl4 wl = unproject_add64(C, dl, L1);
    dbl4 wr = unproject_add64(C, dr, L1);
    Prim64 pl, pr;
    bool ok = pos64(wl.x) && pos64(wr.x);
    if (ok) {
        pl = prim64(wl, gm1);
        pr = prim64(wr, gm1);
        ok = pos64(pl.p) && pos64(pr.p);
    }
    if (!ok) {  // positivity fallback: first-order end states
        wl = L1;
        wr = R1;
        pl = prim64(L1, gm1);
        pr = prim64(R1, gm1);
        atomicAdd(A.fallback, 1ull);
    }

    // Roe flux with Harten's entropy fix (delta = 0.1 c), in the one-sided
    // form F_L + R diag((lambda - |lambda|)/2) L (w_R - w_L): equal to
    // (F_L + F_R)/2 - R |Lambda| L (w_R - w_L)/2 because the Roe matrix
    // satisfies F_R - F_L = R Lambda L (w_R - w_L)
    const Roe64 Q = roe64(wl, pl, wr, pr, nx, ny, gm1, hgm1);
    const dbl4 a = project64(Q, sub4(wr, wl));
    // (l - |l|_fixed) / 2 is min(l, 0) where |l| >= delta and, where Harten's
    // |l|_fixed = (l^2 + delta^2) / (2 delta) applies, -(l - delta)^2 / (4 delta).
    // Both tests run on the integer pipe: |l| < delta compares the bit
    // patterns of two non-negative doubles (delta = 0.1 c is positive), and
    // a NaN l is passed through as the FP64 form would.
    const double delta = 0.1 * Q.c, h4d = 2.5 * Q.ic;  // 1 / (4 delta)
    const unsigned long long dbits = (unsigned long long)__double_as_longlong(delta);
    auto neg = [&](double l) {
        const long long b = __double_as_longlong(l);
        const unsigned long long ab = (unsigned long long)b & 0x7FFFFFFFFFFFFFFFULL;
        if (ab < dbits) {
            const double s = l - delta;
            return -(s * s) * h4d;
        }
        return (b < 0 || ab > 0x7FF0000000000000ULL) ? l : 0.0;
    };
    const double nu = neg(Q.qn), nm = neg(Q.qn - Q.c), np = neg(Q.qn + Q.c);
    const dbl4 D = unproject64(Q, dbl4_make(nm * a.x, nu * a.y, nu * a.z, np * a.w));
    const double qnl = (wl.y * nx + wl.z * ny) * pl.ir;
    dbl4 f;
    f.x = fma(wl.x, qnl, D.x);
    f.y = fma(wl.y, qnl, fma(pl.p, nx, D.y));
    f.z = fma(wl.z, qnl, fma(pl.p, ny, D.z));
    f.w = fma(wl.w + pl.p, qnl, D.w);
    return f;
}
__device__ __forceinline__ void edge_flux_f64_body(const EdgeArgs &A, const int64_t e) {
    st4(static_cast<double *>(A.r), e, edge_flux_f64_value(A, e));
}
// Precision 64 off the double-word path, out of line so that its registers do
// not weigh on that path: the flux r in FP64 (a stage that runs in FP64
// throughout), or its increment r - F_n(L1) as the double words the folded
// divergence reads (a single edge).
__device__ __noinline__ void edge_flux_f64_cold(const EdgeArgs *A, const int64_t e, const bool increment) {
    dbl4 f = edge_flux_f64_value(*A, e);
    if (increment) {
        const dbl4 L1 = ld4v(static_cast<const double *>(A->w), __ldg(A->sten + 2 * A->ne + e));
        const double *coef = static_cast<const double *>(A->coef);
        const double nx = __ldg(coef + (int64_t)kCoefN * A->ne + e), ny = __ldg(coef + (int64_t)(kCoefN + 1) * A->ne + e);
        const Prim64 P = prim64(L1, A->gm1);
        const double mn = fma(L1.y, nx, L1.z * ny), q = mn * P.ir;
        using namespace dwa;
        const dw x = d2dw(f.x - mn), y = d2dw(f.y - fma(L1.y, q, P.p * nx)), z = d2dw(f.z - fma(L1.z, q, P.p * ny)),
                 w = d2dw(f.w - (L1.w + P.p) * q);
        float4 *r = static_cast<float4 *>(A->r);
        r[2 * e] = make_float4(x.h, x.l, y.h, y.l);
        r[2 * e + 1] = make_float4(z.h, z.l, w.h, w.l);
        return;
    }
    st4(static_cast<double *>(A->r), e, f);
}
__device__ __forceinline__ bool stage_is_wide(const int *wide, int in) {
    return (__ldcg(wide + in) | __ldcg(wide + kWideGhost)) != 0;
}
// The flag of vertex v's mesh, where any mesh's is set (through L1: no launch
// writes the slot that it reads).
template <class Args>
__device__ __forceinline__ bool mesh_is_wide(const Args &A, int64_t v) {
    return __ldca(A.wide + kWideSlots * (1 + __ldg(A.wcomp + v)) + A.wide_in) != 0;
}
__device__ __forceinline__ void set_wide(int *wide, const int32_t *wcomp, int64_t v, int slot) {
    wide[slot] = 1;
    if (wcomp) wide[kWideSlots * (1 + __ldg(wcomp + v)) + slot] = 1;
}
// Which meshes' stages are out of the window.
enum Wide { kNone, kAll, kSome };
template <class Args>
__device__ __forceinline__ Wide wide_stage(const Args &A) {
    return !stage_is_wide(A.wide, A.wide_in) ? kNone : A.wcomp ? kSome : kAll;
}
// The same, telling whether all of a batch's are, which spares every edge and
// vertex the look at its mesh's flag (6 meshes, 167k vertices, all outside: 1984
// to 1885 us a step); every thread of the block calls it.
__device__ __forceinline__ Wide wide_batch_stage(const EdgeArgs &A) {
    Wide k = wide_stage(A);
    if (k != kSome) return k;
    int all = 1;
    for (int c = threadIdx.x; c < A.n_comp; c += blockDim.x) all &= __ldcg(A.wide + kWideSlots * (1 + c) + A.wide_in);
    return __syncthreads_and(all) ? kAll : kSome;
}
// One edge at precision 64.
__device__ __forceinline__ void edge_flux_guard_body(const EdgeArgs &A, const int64_t e, const dwa::Stage &S,
                                                     const Wide k) {
    if (k == kAll || (k == kSome && mesh_is_wide(A, __ldg(A.sten + 2 * A.ne + e)))) edge_flux_f64_cold(&A, e, false);
    else if (!dwa::edge_flux_dw_body<true>(A, e, S)) edge_flux_f64_cold(&A, e, true);
}
// A state outside the double words' window: density or energy not in
// [2^-kWideExp, 2^kWideExp), by the exponent field (NaN, zero, negative and
// infinite values fail), or a pressure p that is not positive (the momentum then
// has |m|^2 < 2 rho E, so it is in range too; a NaN or infinite one gives a NaN or
// -infinite pressure).
__device__ __forceinline__ bool outside_window(const dbl4 &w, double p) {
    const unsigned lo = (unsigned)(1023 - kWideExp) << 20, n = (unsigned)(2 * kWideExp) << 20;
    return (unsigned)__double2hiint(w.x) - lo >= n || (unsigned)__double2hiint(w.w) - lo >= n || !pos64(p);
}

// ------------------------------------------------------------------ vertex fluxes
// f, g of a state from its primitives (1/rho, p): the same quantities the
// Roe record needs, so the two share one reciprocal square root.
__device__ __forceinline__ void euler_fg(const dbl4 &w, const Prim64 &P, dbl4 &f, dbl4 &g) {
    const double u = w.y * P.ir, v = w.z * P.ir;
    f = dbl4_make(w.y, fma(w.y, u, P.p), w.z * u, (w.w + P.p) * u);
    g = dbl4_make(w.z, w.y * v, fma(w.z, v, P.p), (w.w + P.p) * v);
}
// Roe-weighted record of a state: (s, s u, s v, s H) with s = sqrt(rho),
// computed with the same operations roe64 applies to each side.
__device__ __forceinline__ dbl4 roe_record64(const dbl4 &w, const Prim64 &P) {
    return dbl4_make(w.x * P.r, w.y * P.r, w.z * P.r, (w.w + P.p) * P.r);
}

__global__ void vertex_flux_f64_kernel(const double *__restrict__ w, double *__restrict__ F, double *__restrict__ Q,
                                       int64_t n, double gm1, int *wide, int64_t n_real, const int32_t *wcomp) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const dbl4 s = ld4(w, v);
    const Prim64 P = prim64(s, gm1);
    dbl4 f, g;
    euler_fg(s, P, f, g);
    st4(F, 2 * v, f);
    st4(F, 2 * v + 1, g);
    if (Q) st4(Q, v, roe_record64(s, P));
    if (wide && outside_window(s, P.p)) set_wide(wide, wcomp, v, v < n_real ? 0 : kWideGhost);
}

// Forward-Euler part of an SSP-RK3 stage, fe = ws + theta dt L.  Without
// the safeguard theta = 1.  With it (alpha > 0), theta is the largest of
// 1, 1/2, ..., 2^-20 (else 0) with rho(fe) >= alpha rho(ws) and
// p(fe) >= alpha p(ws), so that the stage combination of w_n and fe stays
// physical (the set of physical states is convex).
__device__ __forceinline__ dbl4 forward_euler(const dbl4 &ws, const dbl4 &L, double dt, double gm1, double alpha,
                                             unsigned long long *limited) {
    dbl4 fe = dbl4_make(fma(dt, L.x, ws.x), fma(dt, L.y, ws.y), fma(dt, L.z, ws.z), fma(dt, L.w, ws.w));
    if (alpha > 0.0) {
        auto pres = [&](const dbl4 &q) { return gm1 * (q.w - 0.5 * (q.y * q.y + q.z * q.z) / q.x); };
        const double ps = pres(ws);
        double th = 1.0;
        bool ok = false;
        for (int k = 0; k <= 20; ++k) {
            fe = dbl4_make(fma(th * dt, L.x, ws.x), fma(th * dt, L.y, ws.y), fma(th * dt, L.z, ws.z),
                           fma(th * dt, L.w, ws.w));
            if (fe.x >= alpha * ws.x && pres(fe) >= alpha * ps) {
                ok = true;
                break;
            }
            th *= 0.5;
        }
        if (!ok) {
            th = 0.0;
            fe = ws;
        }
        if (th < 1.0) atomicAdd(limited, 1ull);
    }
    return fe;
}

// Two adjacent float4 (record j of a [n][2] float4 buffer: FP32 vertex fluxes
// (f, g), or an edge's double-word increments) as one 32-byte load; the
// buffers are 32-byte aligned and read-only in the kernel.
__device__ __forceinline__ void ld_fg32(const float4 *F, int64_t j, float4 &f, float4 &g) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(f.x), "=f"(f.y), "=f"(f.z), "=f"(f.w), "=f"(g.x), "=f"(g.y), "=f"(g.z), "=f"(g.w)
        : "l"(F + 2 * j));
}

// ------------------------------------------------------------------ FP64 divergence (+ RK stage)
// Position i of the SELL tables; the vertex it holds is A.perm[i].  With
// DWE (precision 48) the edge entries are double-word increments
// r_k - F_n(L1_k) with double-word weights, summed in double words (terms of
// the size of the increments), and the vertex weights carry the folded
// F_n(L1_k) parts.
// Loads of the FP64 / precision-48 divergence tables: read once per stage,
// so in the stage modes they do not allocate in L1 (which keeps it for the
// flux gathers) and each miss asks L2 for 256 bytes; precision-48 divergence
// 0.1435 -> 0.1385 ms at 250k vertices, the FP64 one (FP64-pipe bound)
// unchanged.
template <int MODE> __device__ __forceinline__ int32_t tld(const int32_t *p) {
    if (MODE == 0) return __ldg(p);
    int32_t v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
template <int MODE> __device__ __forceinline__ double tld(const double *p) {
    if (MODE == 0) return __ldg(p);
    double v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.f64 %0, [%1];" : "=d"(v) : "l"(p));
    return v;
}
template <int MODE> __device__ __forceinline__ float2 tld(const float2 *p) {
    if (MODE == 0) return __ldg(p);
    float2 v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
// With LPV > 1 that many consecutive lanes share a position: lane q of them
// takes every LPV-th entry, the partial sums meet by shuffles (every lane of the
// warp calls it, `on` where its position exists) and lane 0 goes on.
template <int MODE, bool DWE = false, int LPV = 1>
__device__ __forceinline__ void div_f64_body(const DivArgs &A, const int64_t i, const int q = 0, const bool on = true) {
    const int64_t sl = on ? i / kSell : 0;
    const int lane = (int)(i % kSell) + q * kSell;
    const int64_t v = !on ? 0 : A.perm ? (int64_t)__ldg(A.perm + i) : i;
    const double *__restrict__ F = static_cast<const double *>(A.F);
    const double *__restrict__ r = static_cast<const double *>(A.r);
    const double *__restrict__ wf = DWE ? A.wf48 : static_cast<const double *>(A.wf);
    const double *__restrict__ wg = DWE ? A.wg48 : static_cast<const double *>(A.wg);
    const double *__restrict__ we = static_cast<const double *>(A.we);
    dbl4 acc = dbl4_make(0, 0, 0, 0);
    {
        const int64_t b = __ldg(A.slice_voff + sl) + lane, e = on ? __ldg(A.slice_voff + sl + 1) : 0;
#pragma unroll 4
        for (int64_t p = b; p < e; p += LPV * kSell) {
            const int32_t j = tld<MODE>(A.vid + p);
            const double a = tld<MODE>(wf + p), c = tld<MODE>(wg + p);
            const dbl4 f = ld4v(F, 2 * (int64_t)j), g = ld4v(F, 2 * (int64_t)j + 1);
            acc.x = fma(a, f.x, fma(c, g.x, acc.x));
            acc.y = fma(a, f.y, fma(c, g.y, acc.y));
            acc.z = fma(a, f.z, fma(c, g.z, acc.z));
            acc.w = fma(a, f.w, fma(c, g.w, acc.w));
        }
    }
    if (DWE) {
        using namespace dwa;
        const float2 *__restrict__ we2 = A.we48;
        const float4 *__restrict__ rd = static_cast<const float4 *>(A.r);
        dot2 sx{0.0f, 0.0f}, sy = sx, sz = sx, sw = sx;
        const int64_t b = __ldg(A.slice_eoff + sl) + lane, e = on ? __ldg(A.slice_eoff + sl + 1) : 0;
#pragma unroll 6
        for (int64_t p = b; p < e; p += LPV * kSell) {
            const int32_t k = tld<MODE>(A.eid + p);
            const float2 wq = tld<MODE>(we2 + p);
            const dw a = dw_make(wq.x, wq.y);
            float4 q0, q1;
            ld_fg32(rd, k, q0, q1);  // the edge's two double-word float4, one 32-byte load
            dot2_add(sx, a, dw_make(q0.x, q0.y));
            dot2_add(sy, a, dw_make(q0.z, q0.w));
            dot2_add(sz, a, dw_make(q1.x, q1.y));
            dot2_add(sw, a, dw_make(q1.z, q1.w));
        }
        const dw rx = dot2_result(sx), ry = dot2_result(sy), rz = dot2_result(sz), rw = dot2_result(sw);
        acc.x += dw2d(rx);
        acc.y += dw2d(ry);
        acc.z += dw2d(rz);
        acc.w += dw2d(rw);
    } else {
        const int64_t b = __ldg(A.slice_eoff + sl) + lane, e = on ? __ldg(A.slice_eoff + sl + 1) : 0;
#pragma unroll 4
        for (int64_t p = b; p < e; p += LPV * kSell) {
            const int32_t k = tld<MODE>(A.eid + p);
            const double a = tld<MODE>(we + p);
            const dbl4 s = ld4v(r, k);
            acc.x = fma(a, s.x, acc.x);
            acc.y = fma(a, s.y, acc.y);
            acc.z = fma(a, s.z, acc.z);
            acc.w = fma(a, s.w, acc.w);
        }
    }
    if (LPV > 1) {
#pragma unroll
        for (int o = 1; o < LPV; o <<= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
            acc.z += __shfl_xor_sync(0xffffffffu, acc.z, o);
            acc.w += __shfl_xor_sync(0xffffffffu, acc.w, o);
        }
        if (q != 0 || !on) return;
    }
    {
        const double *cfg = DWE ? A.cfg48 : static_cast<const double *>(A.cfg);
        const double cf = __ldg(cfg + v), cg = __ldg(cfg + A.n_real + v);
        const dbl4 f = ld4v(F, 2 * v), g = ld4v(F, 2 * v + 1);
        acc.x = fma(cf, f.x, fma(cg, g.x, acc.x));
        acc.y = fma(cf, f.y, fma(cg, g.y, acc.y));
        acc.z = fma(cf, f.z, fma(cg, g.z, acc.z));
        acc.w = fma(cf, f.w, fma(cg, g.w, acc.w));
    }
    const dbl4 L = neg4(acc);  // dw/dt = -(a1 + b2)
    if (MODE == 0) {
        const int64_t row = A.out_map ? (int64_t)__ldg(A.out_map + v) : v;
        st4(A.out, row, L);
        return;
    }
    const double dt = A.comp ? __ldg(A.dt_comp + __ldg(A.comp + v)) : (A.dt_dev ? *A.dt_dev : A.dt);
    const dbl4 ws = ld4v(A.ws, v);
    const dbl4 fe = forward_euler(ws, L, dt, A.gm1, A.pos_alpha, A.limited);
    dbl4 o;
    if (MODE == 1) {
        o = fe;
    } else {
        const dbl4 wn = ld4v(A.wn, v);
        const double cn = MODE == 2 ? 0.75 : 1.0 / 3.0;
        const double cs = MODE == 2 ? 0.25 : 2.0 / 3.0;
        o.x = fma(cn, wn.x, cs * fe.x);
        o.y = fma(cn, wn.y, cs * fe.y);
        o.z = fma(cn, wn.z, cs * fe.z);
        o.w = fma(cn, wn.w, cs * fe.w);
    }
    st4(A.wout, v, o);
    const Prim64 P = prim64(o, A.gm1);
    dbl4 f, g;
    euler_fg(o, P, f, g);
    double *Fo = static_cast<double *>(A.Fout);
    st4(Fo, 2 * v, f);
    st4(Fo, 2 * v + 1, g);
    if (A.Qout) st4(A.Qout, v, roe_record64(o, P));
    if (A.wide && outside_window(o, P.p)) set_wide(A.wide, A.wcomp, v, A.wide_out);
}
// The FP64 form out of line, for the kernels that seldom take it.  It shares a
// vertex between the same lanes: RK3 step outside the window with one of them at
// work / all / in the FP64 kernels alone, one lane to a vertex: 10,000 vertices
// 238 / 163 / 186 us, 22,500 347 / 294 / 294, 55,225 719 / 610 / 578 (the stage
// update of one lane in two takes a warp's FP64 time; a vertex to each thread of
// half the block gives 606 there, and 240 for 222 us at 14,400).
template <int MODE, int LPV>
__device__ __noinline__ void div_f64_cold(const DivArgs *A, const int64_t i, const int q, const bool on) {
    div_f64_body<MODE, false, LPV>(*A, i, q, on);
}
// The divergence of one vertex by KIND (kDivPlain, kDivDw, kDivGuard).  Lanes that
// share a warp but not a mesh take one form after the other, each with the
// other's lanes off.
template <int MODE, int KIND, int LPV = 1>
__device__ __forceinline__ void div_f64_any(const DivArgs &A, const int64_t i, const Wide k, const int q = 0,
                                            bool on = true) {
    if (KIND == kDivGuard && k != kNone) {
        const bool wide = on && (k == kAll || mesh_is_wide(A, A.perm ? (int64_t)__ldg(A.perm + i) : i));
        if (LPV == 1 ? wide : __any_sync(0xffffffffu, wide)) div_f64_cold<MODE, LPV>(&A, i, q, wide);
        on = on && !wide;
        if (LPV == 1 ? !on : !__any_sync(0xffffffffu, on)) return;
    }
    div_f64_body<MODE, KIND != kDivPlain, LPV>(A, i, q, on);
}

// ================================================================== FP32 path
// The FP32 residual reads an FP32 copy of the state and, per edge, the
// FP64-built NU-WENO5 block rounded to FP32 (104 bytes), or in the compact
// form (mesh option f32_coef = 1) the edge's four stencil gaps and normal
// (24 bytes), from which it forms the coefficients in registers; weights,
// fluxes and sums are FP32.  Reciprocals use the hardware approximation
// (rcp.approx, about one ulp), well inside the FP32 path's error against
// FP64.
__device__ __forceinline__ float rcp32(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Read-once loads of the streamed edge tables (the FP32 coefficient block or
// gaps): they do not allocate in L1, which keeps its capacity for the state
// gathers (edge kernel 0.031 -> 0.0275 ms at 250k vertices).
__device__ __forceinline__ float4 ld_stream4(const float4 *p) {
    float4 v;
    asm("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p));
    return v;
}
__device__ __forceinline__ float4 sub4f(float4 a, float4 b) {
    return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
}
__device__ __forceinline__ float4 add4f(float4 a, float4 b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

struct Prim32 {
    float r, ir, p;
};
__device__ __forceinline__ Prim32 prim32(const float4 &w, float gm1) {
    Prim32 q;
    q.r = rsqrtf(w.x);
    q.ir = q.r * q.r;
    q.p = gm1 * (w.w - 0.5f * (w.y * w.y + w.z * w.z) * q.ir);
    return q;
}
struct Roe32 {
    float u, v, H, c, ic, b1h, ich, qn, qt, hq2, nx, ny;  // b1h = b1 / 2, ich = ic / 2
};
__device__ __forceinline__ Roe32 roe32(const float4 &a, const Prim32 &pa, const float4 &b, const Prim32 &pb, float nx,
                                      float ny, float gm1) {
    Roe32 R;
    const float sa = a.x * pa.r, sb = b.x * pb.r;
    const float inv = rcp32(sa + sb);
    R.u = (a.y * pa.r + b.y * pb.r) * inv;
    R.v = (a.z * pa.r + b.z * pb.r) * inv;
    R.H = ((a.w + pa.p) * pa.r + (b.w + pb.p) * pb.r) * inv;
    R.hq2 = 0.5f * (R.u * R.u + R.v * R.v);
    const float c2 = gm1 * (R.H - R.hq2);
    R.ic = rsqrtf(c2);
    R.c = c2 * R.ic;
    R.b1h = 0.5f * gm1 * R.ic * R.ic;
    R.ich = 0.5f * R.ic;
    R.nx = nx;
    R.ny = ny;
    R.qn = R.u * nx + R.v * ny;
    R.qt = R.v * nx - R.u * ny;
    return R;
}
// pre-halved factors (phi/2, psi/2) and the sum started from d.w
__device__ __forceinline__ float4 project32(const Roe32 &R, const float4 &d) {
    const float phh = R.b1h * fmaf(-R.v, d.z, fmaf(-R.u, d.y, fmaf(R.hq2, d.x, d.w)));
    const float psh = (R.qn * d.x - R.nx * d.y - R.ny * d.z) * R.ich;
    return make_float4(phh + psh, fmaf(-2.0f, phh, d.x), R.nx * d.z - R.ny * d.y - R.qt * d.x, phh - psh);
}
__device__ __forceinline__ float4 unproject32(const Roe32 &R, const float4 &c) {
    const float rho = c.x + c.y + c.w;
    const float dd = R.c * (c.w - c.x);
    return make_float4(rho, R.u * rho + R.nx * dd - R.ny * c.z, R.v * rho + R.ny * dd + R.nx * c.z,
                       R.H * (c.x + c.w) + R.hq2 * c.y + R.qn * dd + R.qt * c.z);
}
// base + unproject32(R, c), with base taken into the fused multiply-adds
__device__ __forceinline__ float4 unproject_add32(const Roe32 &R, const float4 &c, const float4 &base) {
    const float ac = c.x + c.w;
    const float rho = ac + c.y;
    const float dd = R.c * (c.w - c.x);
    return make_float4(base.x + rho, fmaf(R.u, rho, fmaf(R.nx, dd, fmaf(-R.ny, c.z, base.y))),
                       fmaf(R.v, rho, fmaf(R.ny, dd, fmaf(R.nx, c.z, base.z))),
                       fmaf(R.H, ac, fmaf(R.hq2, c.y, fmaf(R.qn, dd, fmaf(R.qt, c.z, base.w)))));
}

// FP32 NU-WENO5 increments of one field, both sides (same sub-stencil
// sharing and block layout as weno_pair64_l1).  Weights alpha_k = C_k /
// (beta_k + eps32), omega = alpha / sum(alpha); the four reciprocals of
// (beta + eps32) serve both sides (a product form would underflow in FP32).
__device__ __forceinline__ void weno_pair32(const float *k, float a, float b, float c, float d, float e, float f,
                                            float eps, float &dl, float &dr) {
    const float b2 = b * b, c2 = c * c;
    const float va = fmaf(k[0], a, k[1] * b), vb = fmaf(k[5], b, k[6] * c);
    const float vc = fmaf(k[10], c, k[11] * d), vd = fmaf(k[15], e, k[16] * f);
    const float ia = rcp32(fmaf(k[2], a * a, fmaf(k[3], a * b, fmaf(k[4], b2, eps))));
    const float ib = rcp32(fmaf(k[7], b2, fmaf(k[8], b * c, fmaf(k[9], c2, eps))));
    const float ic = rcp32(fmaf(k[12], c2, fmaf(k[13], c * d, fmaf(k[14], d * d, eps))));
    const float id = rcp32(fmaf(k[17], e * e, fmaf(k[18], e * f, fmaf(k[19], f * f, eps))));
    // middle linear weights are 1 (the block stores C_0/C_1, C_2/C_1);
    // right increments from L1 (S_d's value shifted by +c), as in the FP64 kernel
    const float l0 = k[20] * ia, l1 = ib, l2 = k[21] * ic;
    dl = fmaf(l0, va, fmaf(l1, vb, l2 * vc)) * rcp32(l0 + l1 + l2);
    const float r0 = k[22] * id, r1 = ic, r2 = k[23] * ib;
    dr = fmaf(r0, vd + c, fmaf(r1, vc, r2 * vb)) * rcp32(r0 + r1 + r2);
}

// NU-WENO5 coefficients of one edge in FP32 (Appendix: the sub-stencil
// interpolants' values at the midpoint, their smoothness indicators, and
// the linear weights that make the combination the degree-4 interpolant,
// Eq. S5), in the order of the coefficient block (fdu_internal.h), from
// the four gaps between consecutive stencil points along the curve, each
// divided by the arc length L1-R1:
//   a = L1-L2, b = L2-L3, c = R1-R2, d = R2-R3,
// so that the left side's points are -(1/2+a+b), -(1/2+a), -1/2, 1/2,
// 1/2+c and the right side's (mirrored) the same with (a, b, c) -> (c, d,
// a).  A sub-stencil's Lagrange basis value at 0 of a point x_j is
// x_a x_b / ((x_j - x_a)(x_j - x_b)) over its other two points, its slope
// -(x_a + x_b) / (...) and its curvature 2 / (...); the smoothness
// indicator (slope)^2 + (13/12)(2 curvature)^2 (unit spacing between L1
// and R1) is kept as the quadratic form of the two differences.  The
// linear weights have the closed forms
//   C_0 = (1/2)(1/2+c) / ((1+a+b)(1+a+b+c)),
//   C_2 = (1/2+a+b)(1/2+a) / ((1+a+b+c)(1+a+c)),   C_1 = 1 - C_0 - C_2
// (ratios of degree-4 and sub-stencil Lagrange values), of which the block
// keeps C_0/C_1 and C_2/C_1.  Every factor is a sum of positive gaps, so
// no step cancels.
constexpr float kT3 = 13.0f / 3.0f;  // (13/12) x 2^2
// outer sub-stencil of a side (points -(1/2+a+b), -(1/2+a), -1/2): values
// of its two outer points' differences and the indicator's form
__device__ __forceinline__ void weno_outer32(float a, float b, float *k) {
    const float ab = a + b;
    const float r0 = rcp32(b * ab), r1 = -rcp32(a * b);
    const float s0 = 1.0f + a, s1 = 1.0f + ab;
    k[0] = 0.5f * (0.5f + a) * r0;
    k[1] = 0.5f * (0.5f + ab) * r1;
    k[2] = r0 * r0 * fmaf(s0, s0, kT3);
    k[3] = 2.0f * r0 * r1 * fmaf(s0, s1, kT3);
    k[4] = r1 * r1 * fmaf(s1, s1, kT3);
}
// C_0/C_1 and C_2/C_1 of a side from its gaps (a, b) and the far side's c
__device__ __forceinline__ void weno_ratios32(float a, float b, float c, float *k) {
    const float p = 1.0f + a + b, r = 1.0f + a + c;
    const float n0r = 0.5f * (0.5f + c) * r, n2p = (0.5f + a + b) * (0.5f + a) * p;
    const float ir = rcp32((p + c) * p * r - n0r - n2p);
    k[0] = n0r * ir;
    k[1] = n2p * ir;
}
__device__ __forceinline__ void weno_coef32(const float4 g, float *k) {
    const float a = g.x, b = g.y, c = g.z, d = g.w;
    weno_outer32(a, b, k);  // S_a
    {                       // S_b: points -(1/2+a), -1/2, 1/2
        const float r2 = rcp32(1.0f + a), r0 = rcp32(a * (1.0f + a));
        k[5] = -0.25f * r0;
        k[6] = 0.5f * (0.5f + a) * r2;
        k[7] = kT3 * r0 * r0;
        k[8] = 2.0f * kT3 * r0 * r2;
        k[9] = fmaf(kT3 * r2, r2, 1.0f);
    }
    {  // S_c: points -1/2, 1/2, 1/2+c
        const float r1 = -rcp32(c), r2 = rcp32(c * (1.0f + c));
        k[10] = -0.5f * (0.5f + c) * r1;
        k[11] = -0.25f * r2;
        k[12] = fmaf(kT3 * r1, r1, 1.0f);
        k[13] = 2.0f * kT3 * r1 * r2;
        k[14] = kT3 * r2 * r2;
    }
    weno_outer32(c, d, k + 15);  // S_d
    weno_ratios32(a, b, c, k + kCoefCL);
    weno_ratios32(c, d, a, k + kCoefCR);
}

// GAPS: the compact coefficient form (the values formed here from the
// edge's stencil gaps); otherwise the FP64-built block rounded to FP32.
template <bool GAPS>
__device__ __forceinline__ void edge_flux_f32_body(const EdgeArgs &A, const int64_t e) {
    const float4 *__restrict__ w = static_cast<const float4 *>(A.w);
    const float *__restrict__ g = static_cast<const float *>(A.coef);
    const float gm1 = A.gm1f;
    const float eps = A.epsf;
    const int64_t ne = A.ne;
    int32_t s[6];
    // the stencil ids are read once as well (the divergence that follows gains
    // more than this kernel loses: 0.055 -> 0.0537 against 0.0275 -> 0.0283 ms)
#pragma unroll
    for (int i = 0; i < 6; ++i)
        asm("ld.global.nc.L1::no_allocate.b32 %0, [%1];" : "=r"(s[i]) : "l"(A.sten + (int64_t)i * ne + e));
    float k[kCoefN];
    float nx, ny;
    if (GAPS) {
        // the edge's stencil gaps ([ne] float4) and normal ([ne] float2 after them)
        const float2 nq = __ldg(reinterpret_cast<const float2 *>(g + (int64_t)4 * ne) + e);
        nx = nq.x;
        ny = nq.y;
        weno_coef32(ld_stream4(reinterpret_cast<const float4 *>(g) + e), k);
    } else {
        // six float4 of values ([c/4][ne] float4, component c%4), then the
        // normal as one float2 ([ne] float2 after them)
        const float4 *__restrict__ g4 = reinterpret_cast<const float4 *>(g);
#pragma unroll
        for (int i = 0; i < kEdgeCoef32Vec; ++i) {
            const float4 q = ld_stream4(g4 + (int64_t)i * ne + e);
            k[4 * i] = q.x;
            k[4 * i + 1] = q.y;
            k[4 * i + 2] = q.z;
            k[4 * i + 3] = q.w;
        }
        const float2 nq = __ldg(reinterpret_cast<const float2 *>(g + (int64_t)4 * kEdgeCoef32Vec * ne) + e);
        nx = nq.x;
        ny = nq.y;
    }
    const float4 L1 = __ldg(w + s[2]), R1 = __ldg(w + s[3]);
    const Prim32 pL1 = prim32(L1, gm1), pR1 = prim32(R1, gm1);
    const Roe32 C = roe32(L1, pL1, R1, pR1, nx, ny, gm1);
    const float4 cM = project32(C, sub4f(R1, L1));
    const float4 cL2 = project32(C, sub4f(__ldg(w + s[1]), L1));
    const float4 cL3 = project32(C, sub4f(__ldg(w + s[0]), L1));
    const float4 cR2 = project32(C, sub4f(__ldg(w + s[4]), R1));
    const float4 cR3 = project32(C, sub4f(__ldg(w + s[5]), R1));
    const float4 cR2L = add4f(cR2, cM);
    float4 dl, dr;
    weno_pair32(k, cL3.x, cL2.x, cM.x, cR2L.x, cR3.x, cR2.x, eps, dl.x, dr.x);
    weno_pair32(k, cL3.y, cL2.y, cM.y, cR2L.y, cR3.y, cR2.y, eps, dl.y, dr.y);
    weno_pair32(k, cL3.z, cL2.z, cM.z, cR2L.z, cR3.z, cR2.z, eps, dl.z, dr.z);
    weno_pair32(k, cL3.w, cL2.w, cM.w, cR2L.w, cR3.w, cR2.w, eps, dl.w, dr.w);

    float4 wl = unproject_add32(C, dl, L1);
    float4 wr = unproject_add32(C, dr, L1);
    Prim32 pl, pr;
    bool ok = wl.x > 0.f && wr.x > 0.f;
    if (ok) {
        pl = prim32(wl, gm1);
        pr = prim32(wr, gm1);
        ok = pl.p > 0.f && pr.p > 0.f;
    }
    if (!ok) {
        wl = L1;
        wr = R1;
        pl = pL1;
        pr = pR1;
        atomicAdd(A.fallback, 1ull);
    }
    // one-sided Roe flux F_L + R diag((lambda - |lambda|)/2) L (w_R - w_L)
    const Roe32 Q = roe32(wl, pl, wr, pr, nx, ny, gm1);
    const float4 a = project32(Q, sub4f(wr, wl));
    const float delta = 0.1f * Q.c, h2d = 5.0f * Q.ic;
    auto neg = [&](float l) {
        const float m = fabsf(l);
        return 0.5f * (l - (m < delta ? fmaf(l, l, delta * delta) * h2d : m));
    };
    const float nu = neg(Q.qn), nm = neg(Q.qn - Q.c), np = neg(Q.qn + Q.c);
    const float4 D = unproject32(Q, make_float4(nm * a.x, nu * a.y, nu * a.z, np * a.w));
    const float qnl = (wl.y * nx + wl.z * ny) * pl.ir;
    float4 f;
    f.x = fmaf(wl.x, qnl, D.x);
    f.y = fmaf(wl.y, qnl, fmaf(pl.p, nx, D.y));
    f.z = fmaf(wl.z, qnl, fmaf(pl.p, ny, D.z));
    f.w = fmaf(wl.w + pl.p, qnl, D.w);
    static_cast<float4 *>(A.r)[e] = f;
}

__device__ __forceinline__ void euler_fg32(const float4 &w, float gm1, float4 &f, float4 &g) {
    const float ir = rcp32(w.x);
    const float u = w.y * ir, v = w.z * ir;
    const float p = gm1 * (w.w - 0.5f * (w.y * u + w.z * v));
    f = make_float4(w.y, fmaf(w.y, u, p), w.z * u, (w.w + p) * u);
    g = make_float4(w.z, w.y * v, fmaf(w.z, v, p), (w.w + p) * v);
}

__global__ void vertex_flux_f32_kernel(const double *__restrict__ w, float4 *__restrict__ F, float4 *__restrict__ w32,
                                       int64_t n, float gm1) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= n) return;
    const dbl4 d = ld4(w, v);
    const float4 s = make_float4((float)d.x, (float)d.y, (float)d.z, (float)d.w);
    w32[v] = s;
    float4 f, g;
    euler_fg32(s, gm1, f, g);
    F[2 * v] = f;
    F[2 * v + 1] = g;
}

template <int MODE>
__device__ __forceinline__ void div_f32_finish(const DivArgs &A, const int64_t v, float4 acc) {
    const float4 *__restrict__ F = static_cast<const float4 *>(A.F);
    {
        const float *cfg = static_cast<const float *>(A.cfg);
        const float cf = __ldg(cfg + v), cg = __ldg(cfg + A.n_real + v);
        const float4 f = __ldg(F + 2 * v), g = __ldg(F + 2 * v + 1);
        acc.x = fmaf(cf, f.x, fmaf(cg, g.x, acc.x));
        acc.y = fmaf(cf, f.y, fmaf(cg, g.y, acc.y));
        acc.z = fmaf(cf, f.z, fmaf(cg, g.z, acc.z));
        acc.w = fmaf(cf, f.w, fmaf(cg, g.w, acc.w));
    }
    const dbl4 L = dbl4_make(-(double)acc.x, -(double)acc.y, -(double)acc.z, -(double)acc.w);
    if (MODE == 0) {
        const int64_t row = A.out_map ? (int64_t)__ldg(A.out_map + v) : v;
        st4(A.out, row, L);
        return;
    }
    // SSP-RK3 combination in FP64
    const double dt = A.comp ? __ldg(A.dt_comp + __ldg(A.comp + v)) : (A.dt_dev ? *A.dt_dev : A.dt);
    const dbl4 ws = ld4(A.ws, v);
    const dbl4 fe = forward_euler(ws, L, dt, A.gm1, A.pos_alpha, A.limited);
    dbl4 o;
    if (MODE == 1) {
        o = fe;
    } else {
        const dbl4 wn = ld4(A.wn, v);
        const double cn = MODE == 2 ? 0.75 : 1.0 / 3.0;
        const double cs = MODE == 2 ? 0.25 : 2.0 / 3.0;
        o.x = fma(cn, wn.x, cs * fe.x);
        o.y = fma(cn, wn.y, cs * fe.y);
        o.z = fma(cn, wn.z, cs * fe.z);
        o.w = fma(cn, wn.w, cs * fe.w);
    }
    st4(A.wout, v, o);
    const float4 s32 = make_float4((float)o.x, (float)o.y, (float)o.z, (float)o.w);
    A.w32out[v] = s32;
    float4 f, g;
    euler_fg32(s32, A.gm1f, f, g);
    float4 *Fo = static_cast<float4 *>(A.Fout);
    Fo[2 * v] = f;
    Fo[2 * v + 1] = g;
}

// Loads of the streamed divergence tables: read once per stage, so they do
// not allocate in L1 (which keeps its capacity for the flux gathers), and
// each miss asks L2 for 256 bytes (the row's 128-byte line and the next).
__device__ __forceinline__ int32_t ld_stream(const int32_t *p) {
    int32_t v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_stream(const float *p) {
    float v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
// Table loads of the FP32 divergence: streaming loads in the fused stage
// (modes 1..3: 0.066 -> 0.062 ms at 250k vertices), plain cached loads for
// the residual alone (mode 0, where the streaming form measured slower).
template <int MODE, class T>
__device__ __forceinline__ T ld_table(const T *p) {
    if (MODE != 0) return ld_stream(p);
    return __ldg(p);
}

template <int MODE>
__device__ __forceinline__ void div_f32_body(const DivArgs &A, const int64_t v) {
    const int64_t sl = v / kSell;
    const int lane = (int)(v % kSell);
    const float4 *__restrict__ F = static_cast<const float4 *>(A.F);
    const float4 *__restrict__ r = static_cast<const float4 *>(A.r);
    const float *__restrict__ wf = static_cast<const float *>(A.wf);
    const float *__restrict__ wg = static_cast<const float *>(A.wg);
    const float *__restrict__ we = static_cast<const float *>(A.we);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    {
        const int64_t b = __ldg(A.slice_voff + sl) + lane, e = __ldg(A.slice_voff + sl + 1);
#pragma unroll 4
        for (int64_t p = b; p < e; p += kSell) {
            const int32_t j = ld_table<MODE>(A.vid + p);
            const float a = ld_table<MODE>(wf + p), c = ld_table<MODE>(wg + p);
            float4 f, g;
            ld_fg32(F, j, f, g);
            acc.x = fmaf(a, f.x, fmaf(c, g.x, acc.x));
            acc.y = fmaf(a, f.y, fmaf(c, g.y, acc.y));
            acc.z = fmaf(a, f.z, fmaf(c, g.z, acc.z));
            acc.w = fmaf(a, f.w, fmaf(c, g.w, acc.w));
        }
    }
    {
        const int64_t b = __ldg(A.slice_eoff + sl) + lane, e = __ldg(A.slice_eoff + sl + 1);
#pragma unroll 8
        for (int64_t p = b; p < e; p += kSell) {
            const int32_t k = ld_table<MODE>(A.eid + p);
            const float a = ld_table<MODE>(we + p);
            const float4 q = __ldg(r + k);
            acc.x = fmaf(a, q.x, acc.x);
            acc.y = fmaf(a, q.y, acc.y);
            acc.z = fmaf(a, q.z, acc.z);
            acc.w = fmaf(a, q.w, acc.w);
        }
    }
    div_f32_finish<MODE>(A, v, acc);
}

// ------------------------------------------------------------------ kernels
__global__ void __launch_bounds__(kEdgeBlock) edge_flux_f64_kernel(EdgeArgs A) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= A.ne) return;
    if (A.dt_dev && *A.dt_dev == 0.0) return;  // adaptive run already at t_end
    edge_flux_f64_body(A, e);
}
// compact form: 80 registers, 24 warps per SM; the streamed block: 95 registers
// and 20 warps (at 80 it spills)
template <bool GAPS>
__global__ void __launch_bounds__(kEdgeBlock, GAPS ? 6 : 5) edge_flux_f32_kernel(EdgeArgs A) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= A.ne) return;
    if (A.dt_dev && *A.dt_dev == 0.0) return;  // adaptive run already at t_end
    edge_flux_f32_body<GAPS>(A, e);
}
// Precision 64: the double-word edge flux, or FP64 where the state is outside
// its window or an edge fails its guard (edge_flux_dw_body).  In FP64 throughout
// the kernel is bound by GB300's FP64 pipe (449 instructions per edge, each 64
// cycles of a sub-partition's pipe, 90 % busy): 0.618 ms at 250k vertices, and
// the divergence after it 0.186 ms; on the double-word path 0.119 and 0.128 ms.
// Error of the residual against plain FP64 (vortex 40^2 / Riemann 101^2 / Sod
// 55^2 of degree 5): 2.3e-14 / 6.5e-14 / 2.2e-14 before, 6.9e-15 / 3.4e-15 /
// 1.1e-14 now: the increments are small against the state, and the folded
// weights leave fewer large terms to cancel in the divergence.
__global__ void __launch_bounds__(kEdgeBlock, 4) edge_flux_guard_kernel(const __grid_constant__ EdgeArgs A) {
    __shared__ float4 stage[dwa::kDwSlots * kEdgeBlock];
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= A.ne) return;
    if (A.dt_dev && *A.dt_dev == 0.0) return;
    dwa::clear_wide(A, e);
    edge_flux_guard_body(A, e, dwa::Stage{stage + threadIdx.x, kEdgeBlock}, wide_stage(A));
}
// At most 80 registers (6 blocks, 24 warps per SM): with the 56 the compiler
// takes when left alone fewer gathers are in flight (precision 48 0.139 against
// 0.120 ms at 250k vertices; 64 registers 0.123, 40 with 9 blocks 0.139).
template <int MODE, int KIND, int LPV>
__global__ void __launch_bounds__(kDivBlock, 6) div_f64_kernel(const __grid_constant__ DivArgs A) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / LPV;
    if (LPV == 1 && i >= A.n_real) return;
    if (MODE != 0 && A.dt_dev && *A.dt_dev == 0.0) return;  // adaptive run already at t_end
    div_f64_any<MODE, KIND, LPV>(A, i, KIND == kDivGuard ? wide_stage(A) : kNone,
                                 (int)threadIdx.x % LPV, i < A.n_real);
}
// ------------------------------------------------------------------ divergence tiles
constexpr int kTileThreads = 256;  // threads of the tile-building kernels
constexpr int kTileSteps = 96;     // longest slice whose entries are scheduled over the banks
// The real entries of vertex v in a SELL layout (natural order): J vertex
// entries (padding names v itself, which is never its own neighbour) and K edge
// entries (padding repeats the first).
struct TileRow {
    int64_t vb, eb;
    int J, K;
};
__device__ __forceinline__ TileRow tile_row(const TileSource &S, int64_t v) {
    const int64_t sl = v / kSell;
    const int lane = (int)(v % kSell);
    TileRow r;
    r.vb = S.slice_voff[sl] + lane;
    r.eb = S.slice_eoff[sl] + lane;
    const int64_t ve = S.slice_voff[sl + 1], ee = S.slice_eoff[sl + 1];
    r.J = r.K = 0;
    for (int64_t p = r.vb; p < ve; p += kSell) r.J += S.vid[p] != (int32_t)v;
    for (int64_t p = r.eb; p < ee; p += kSell) r.K += p == r.eb || S.eid[p] != S.eid[r.eb];
    return r;
}
// One tile's shared state while it is built.
struct TileWork {
    union {
        int32_t hash[2 * kTileMaxE];
        unsigned short pos[kTileSteps][kTile];  // a lane's positions in the tile's list, in list order
    };
    int32_t list[kTileMaxE];
    int count;
    int J[kTile], K[kTile];                 // by position
    unsigned char bank[kTileSteps][kTile];  // bank of the entry a lane takes at each step (8: none)
};
// The tile's distinct vertices (edges = false; with the tile's own) or edges:
// a hash table in shared memory, compacted and sorted.  Returns the count, -1
// beyond the capacity.  Every thread of the block calls it.
__device__ int tile_unique(TileWork &W, const TileSource &S, int64_t v0, int nvt, bool edges) {
    const int most = edges ? kTileMaxE : kTileMaxV, cap = 2 * most;
    for (int i = threadIdx.x; i < cap; i += kTileThreads) W.hash[i] = -1;
    if (threadIdx.x == 0) W.count = 0;
    __syncthreads();
    auto insert = [&](int32_t id) {
        unsigned h = ((unsigned)id * 2654435761u) & (unsigned)(cap - 1);
        while (*(volatile int *)&W.count <= most) {  // at most half of the slots are ever taken, plus one per thread
            const int32_t old = atomicCAS(W.hash + h, -1, id);
            if (old == -1) atomicAdd(&W.count, 1);
            if (old == -1 || old == id) break;
            h = (h + 1) & (unsigned)(cap - 1);
        }
    };
    constexpr int kShare = kTileThreads / kTile;  // threads that share a vertex's entries
    const int i0 = threadIdx.x % kTile, j0 = threadIdx.x / kTile;
    if (i0 < nvt) {
        const TileRow r = tile_row(S, v0 + i0);
        if (edges) {
            for (int j = j0; j < r.K; j += kShare) insert(S.eid[r.eb + (int64_t)kSell * j]);
        } else {
            if (j0 == 0) insert((int32_t)(v0 + i0));
            for (int j = j0; j < r.J; j += kShare) insert(S.vid[r.vb + (int64_t)kSell * j]);
        }
    }
    __syncthreads();
    const int total = W.count;
    __syncthreads();
    if (total > most) return -1;
    if (threadIdx.x == 0) W.count = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < cap; i += kTileThreads)
        if (W.hash[i] >= 0) W.list[atomicAdd(&W.count, 1)] = W.hash[i];
    int m = 1;
    while (m < total) m <<= 1;
    __syncthreads();
    for (int i = total + (int)threadIdx.x; i < m; i += kTileThreads) W.list[i] = INT32_MAX;
    __syncthreads();
    for (int k = 2; k <= m; k <<= 1)  // bitonic sort
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < m; i += kTileThreads) {
                const int q = i ^ j;
                if (q > i) {
                    const int32_t a = W.list[i], c = W.list[q];
                    if ((a > c) == ((i & k) == 0)) {
                        W.list[i] = c;
                        W.list[q] = a;
                    }
                }
            }
            __syncthreads();
        }
    return total;
}
__device__ unsigned short tile_position(const int32_t *list, int n, int32_t id) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (list[mid] < id) lo = mid + 1;
        else hi = mid;
    }
    return (unsigned short)lo;
}
// Grid (tiles, 2): vertices and edges of a tile are built by two blocks.  On a
// small mesh the time is one block's serial chain (1600 vertices: the sizes in
// 50 us and the tables in 178, with one block after the other 62 and 262).
__global__ void __launch_bounds__(kTileThreads)
    tile_count_kernel(TileSource S, TileTables T, int32_t *nv, int32_t *ne, int32_t *gv, int32_t *ge) {
    extern __shared__ int tile_work[];
    TileWork &W = *reinterpret_cast<TileWork *>(tile_work);
    __shared__ int key[kTile];
    const int64_t t = blockIdx.x, p0 = t * kTile, v0 = S.start[t];
    const int nvt = S.start[t + 1] - S.start[t], i = threadIdx.x;
    const bool edges = blockIdx.y != 0;
    TileRow r{0, 0, 0, 0};
    if (i < kTile) {
        if (i < nvt) r = tile_row(S, v0 + i);
        key[i] = i < nvt ? (r.J << 16) | r.K : -1;
    }
    __syncthreads();
    if (i < kTile && !edges) {  // decreasing (J, K), ties in vertex order
        int rank = 0;
        for (int q = 0; q < kTile; ++q) rank += key[q] > key[i] || (key[q] == key[i] && q < i);
        W.J[rank] = r.J;
        W.K[rank] = r.K;
        T.perm[p0 + rank] = i < nvt ? (int32_t)(v0 + i) : -1;
    }
    __syncthreads();
    if (i < kTile / kSell && !edges) {
        int mj = 0, mk = 0;
        for (int l = 0; l < kSell; ++l) {
            mj = max(mj, W.J[i * kSell + l]);
            mk = max(mk, W.K[i * kSell + l]);
        }
        gv[t * (kTile / kSell) + i] = (mj + 3) / 4;
        ge[t * (kTile / kSell) + i] = (mk + 3) / 4;
    }
    const int n = tile_unique(W, S, v0, nvt, edges);
    if (i == 0) (edges ? ne : nv)[t] = n;
}
// Order of a slice's entries over its steps.  A 16-byte shared-memory read is
// served eight lanes at a time, and positions equal modulo 8 fall on the same
// banks, so each group of eight lanes takes entries of different banks where it
// can: per step, each lane (starting from another one each time) takes the next
// bank, from its own place in a rotation, that it has entries of and no lane
// before it took; otherwise it waits a step if it has some to spare, or takes
// a taken one.  One thread per group; n[l] = entries of lane l, left[l] = their
// counts by bank, a byte each.
__device__ void tile_schedule(TileWork &W, int group, int steps, const int *n) {
    unsigned long long left[8];
    unsigned has[8];
    int rest[8];
#pragma unroll
    for (int l = 0; l < 8; ++l) {
        left[l] = 0;
        rest[l] = n[8 * group + l];
        for (int j = 0; j < rest[l]; ++j) left[l] += 1ull << (8 * (W.pos[j][8 * group + l] & 7));
        has[l] = 0;
        for (int c = 0; c < 8; ++c) has[l] |= (unsigned)((left[l] >> (8 * c) & 0xff) != 0) << c;
    }
    for (int s0 = 0; s0 < steps; s0 += 8)
#pragma unroll
        for (int ds = 0; ds < 8; ++ds) {
            const int s = s0 + ds;
            if (s >= steps) break;
            unsigned used = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int l = (q + ds) & 7, first = (s + l) & 7;
                unsigned m = has[l] & ~used;
                if (m == 0 && rest[l] >= steps - s) m = has[l];
                int c = 8;
                if (m) {
                    c = (__ffs((m | m << 8) >> first) - 1 + first) & 7;
                    used |= 1u << c;
                    left[l] -= 1ull << (8 * c);
                    if ((left[l] >> (8 * c) & 0xff) == 0) has[l] &= ~(1u << c);
                    --rest[l];
                }
                W.bank[s][8 * group + l] = (unsigned char)c;
            }
        }
}
__global__ void __launch_bounds__(kTileThreads) tile_fill_kernel(TileSource S, TileTables T) {
    extern __shared__ int tile_work[];
    TileWork &W = *reinterpret_cast<TileWork *>(tile_work);
    const int64_t t = blockIdx.x, p0 = t * kTile, v0 = S.start[t];
    const int nvt = S.start[t + 1] - S.start[t], i = threadIdx.x;
    const int32_t v = i < kTile ? T.perm[p0 + i] : -1;
    const TileRow r = v >= 0 ? tile_row(S, v) : TileRow{0, 0, 0, 0};
    const int64_t sl = t * (kTile / kSell) + i / kSell, lane = i % kSell;
    const int part = blockIdx.y;  // 0: vertices, 1: edges
    const int32_t *ids = part ? S.eid : S.vid;
    const int64_t b = part ? r.eb : r.vb;
    const int cnt = part ? r.K : r.J;
    const int32_t *goff = part ? T.geoff : T.gvoff;
    const int n = tile_unique(W, S, v0, nvt, part != 0);
    int32_t *list = part ? T.elist + T.eoff[t] : T.vlist + T.voff[t];
    for (int q = i; q < n; q += kTileThreads) list[q] = W.list[q];
    const int64_t g0 = i < kTile ? goff[sl] : 0;
    const int steps = i < kTile ? 4 * (int)(goff[sl + 1] - g0) : 0;
    const bool scheduled = steps <= kTileSteps;  // the same for the lanes of a slice
    int *count = part ? W.K : W.J;
    __syncthreads();  // the hash table's memory holds positions from here
    if (i < kTile) {
        count[i] = cnt;
        if (scheduled)
            for (int j = 0; j < cnt; ++j) W.pos[j][i] = tile_position(W.list, n, ids[b + (int64_t)kSell * j]);
    }
    __syncthreads();
    if (i < kTile && scheduled && i % 8 == 0) tile_schedule(W, i / 8, steps, count);
    __syncthreads();
    if (i < kTile) {
        // a step without an entry repeats the lane's first with weight 0, as
        // the SELL padding does, so that a non-finite flux reaches only the
        // vertices whose stencils hold it
        unsigned short *pos = reinterpret_cast<unsigned short *>(part ? T.epos : T.vpos);
        float *wa = reinterpret_cast<float *>(part ? T.we : T.wf), *wb = reinterpret_cast<float *>(T.wg);
        const float *sa = part ? S.we : S.wf;
        unsigned char cur[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (int s = 0; s < steps; ++s) {
            int j = s < cnt ? s : -1;
            unsigned short p = 0;
            if (scheduled) {
                const int c = W.bank[s][i];
                j = -1;
                if (c < 8) {
                    j = cur[c];
                    while ((W.pos[j][i] & 7) != c) ++j;
                    cur[c] = (unsigned char)(j + 1);
                }
                if (cnt > 0) p = W.pos[j < 0 ? 0 : j][i];
            } else if (cnt > 0) {
                p = tile_position(W.list, n, ids[b + (int64_t)kSell * (j < 0 ? 0 : j)]);
            }
            const int64_t q = 4 * ((g0 + s / 4) * kSell + lane) + s % 4, src = b + (int64_t)kSell * j;
            pos[q] = p;
            wa[q] = j >= 0 ? sa[src] : 0.0f;
            if (!part) wb[q] = j >= 0 ? S.wg[src] : 0.0f;
        }
    }
}

__device__ __forceinline__ void cp_async16(void *smem, const void *g) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(g)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ ushort4 ld_stream(const ushort4 *p) {
    ushort4 v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.v4.u16 {%0, %1, %2, %3}, [%4];"
        : "=h"(v.x), "=h"(v.y), "=h"(v.z), "=h"(v.w)
        : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld_stream(const float4 *p) {
    float4 v;
    asm("ld.global.nc.L1::no_allocate.L2::256B.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p));
    return v;
}

// FP32 divergence (+ stage) over tiles: one block copies its tile's fluxes into
// shared memory, then each thread walks the entries of one vertex there.
//
// What bounds it: the table stream (about 510 bytes per vertex from DRAM, 60 %
// of the measured HBM rate) and its latency; the reads of the staged fluxes
// take half of the shared-memory cycles.  Gathering every entry from global
// memory (div_f32_kernel) costs 12 L1 wavefronts where 4 would carry the data
// (L1 76 % busy) and 8 and 12 bytes per entry with full ids: 0.0532 ms in the
// stage and 0.066 ms for the residual alone at 250k vertices, here 0.0417 and
// 0.0354 ms.  On the way: the same tables staged 0.050 (16-bit positions),
// entries in groups of four 0.0467, banks scheduled (tile_schedule) 0.0445, 73
// registers and 7 blocks per SM instead of 64 and 8 0.0417.  Tiles of 256
// (0.054), table groups read ahead explicitly (0.044 to 0.064) and 6 or 9
// blocks per SM (0.052, 0.045) are slower.
//
// One tile by kTile threads (tid of them, staging in sm); sync() holds those
// threads until the staging of all is done.
template <int MODE, class Sync>
__device__ __forceinline__ void div_f32_tile_body(const DivArgs &A, const TileTables &T, const int64_t t, const int tid,
                                                  float4 *sm, Sync &&sync) {
    const int v0 = __ldg(T.voff + t), nvt = __ldg(T.voff + t + 1) - v0;
    const int e0 = __ldg(T.eoff + t), net = __ldg(T.eoff + t + 1) - e0;
    float4 *sf = sm, *sg = sm + nvt, *sr = sm + 2 * nvt;
    const float4 *__restrict__ F = static_cast<const float4 *>(A.F);
    const float4 *__restrict__ r = static_cast<const float4 *>(A.r);
    for (int i = tid; i < net; i += kTile) cp_async16(sr + i, r + __ldg(T.elist + e0 + i));
    for (int i = tid; i < nvt; i += kTile) {
        const int64_t j = __ldg(T.vlist + v0 + i);
        cp_async16(sf + i, F + 2 * j);
        cp_async16(sg + i, F + 2 * j + 1);
    }
    const int64_t sl = t * (kTile / kSell) + tid / kSell;
    const int lane = tid % kSell;
    const int32_t v = __ldg(T.perm + t * kTile + tid);
    const int gb = __ldg(T.gvoff + sl), ge = __ldg(T.gvoff + sl + 1);
    const int hb = __ldg(T.geoff + sl), he = __ldg(T.geoff + sl + 1);
    cp_async_wait();
    sync();
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    auto vert = [&](int j, float a, float c) {
        const float4 f = sf[j], g = sg[j];
        acc.x = fmaf(a, f.x, fmaf(c, g.x, acc.x));
        acc.y = fmaf(a, f.y, fmaf(c, g.y, acc.y));
        acc.z = fmaf(a, f.z, fmaf(c, g.z, acc.z));
        acc.w = fmaf(a, f.w, fmaf(c, g.w, acc.w));
    };
#pragma unroll 2
    for (int g = gb; g < ge; ++g) {
        const ushort4 j = ld_stream(T.vpos + (int64_t)g * kSell + lane);
        const float4 a = ld_stream(T.wf + (int64_t)g * kSell + lane), c = ld_stream(T.wg + (int64_t)g * kSell + lane);
        vert(j.x, a.x, c.x);
        vert(j.y, a.y, c.y);
        vert(j.z, a.z, c.z);
        vert(j.w, a.w, c.w);
    }
    auto edge = [&](int k, float a) {
        const float4 q = sr[k];
        acc.x = fmaf(a, q.x, acc.x);
        acc.y = fmaf(a, q.y, acc.y);
        acc.z = fmaf(a, q.z, acc.z);
        acc.w = fmaf(a, q.w, acc.w);
    };
#pragma unroll 4
    for (int h = hb; h < he; ++h) {
        const ushort4 k = ld_stream(T.epos + (int64_t)h * kSell + lane);
        const float4 a = ld_stream(T.we + (int64_t)h * kSell + lane);
        edge(k.x, a.x);
        edge(k.y, a.y);
        edge(k.z, a.z);
        edge(k.w, a.w);
    }
    if (v >= 0) div_f32_finish<MODE>(A, v, acc);
}
template <int MODE>
__global__ void __launch_bounds__(kTile, 7) div_f32_tile_kernel(const __grid_constant__ DivArgs A,
                                                                 const __grid_constant__ TileTables T) {
    extern __shared__ float4 sm[];
    if (MODE != 0 && A.dt_dev && *A.dt_dev == 0.0) return;
    div_f32_tile_body<MODE>(A, T, blockIdx.x, threadIdx.x, sm, [] { __syncthreads(); });
}

// Folded tables of the double-word divergence (launch_fold_tables).  Entries and
// sums in the order of the SELL lists, rounded one by one.  kFoldLanes threads
// serve a SELL position: each takes every kFoldLanes-th vertex entry, sums in
// registers the edges whose left vertex it is, and looks at all of the position's
// edges for that (independent loads).  One thread per position, adding to the
// table for each edge in turn, waited for its own stores: the double-word tables
// of 1600 vertices took 172 us in all, 118 now.
constexpr int kFoldLanes = 8;
__global__ void fold_tables_kernel(DivArgs A, const int32_t *__restrict__ left, const double *__restrict__ nx,
                                   const double *__restrict__ ny, double *wf48, double *wg48, float2 *we48,
                                   double *cfg48, int *bad) {
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / kFoldLanes;
    const int sub = (int)threadIdx.x % kFoldLanes;
    const int64_t sl = i / kSell;
    if (sl >= (A.n_real + kSell - 1) / kSell) return;  // a slice's threads fill whole warps
    const int lane = (int)(i % kSell);
    const int64_t vb = A.slice_voff[sl] + lane, ve = A.slice_voff[sl + 1];
    const int64_t eb = A.slice_eoff[sl] + lane, ee = A.slice_eoff[sl + 1];
    const double *__restrict__ wf = static_cast<const double *>(A.wf), *__restrict__ wg = static_cast<const double *>(A.wg);
    const double *__restrict__ we = static_cast<const double *>(A.we), *__restrict__ cfg = static_cast<const double *>(A.cfg);
    const bool real = i < A.n_real;
    const int32_t v = real ? A.perm[i] : -1;
    int flag = 0, edges = 0, found = 0;
    // f, g += the normals of the edges (not padding) that start at `id`, times their weights
    auto sum = [&](int32_t id, double &f, double &g) {
#pragma unroll 4
        for (int64_t q = eb; q < ee; q += kSell) {
            const double w = we[q];
            const int32_t e = A.eid[q];
            if (w == 0.0 || left[e] != id) continue;
            f = __dadd_rn(f, __dmul_rn(w, nx[e]));
            g = __dadd_rn(g, __dmul_rn(w, ny[e]));
            ++found;
        }
    };
    for (int64_t p = vb + (int64_t)kSell * sub; p < ve; p += kSell * kFoldLanes) {
        double f = wf[p], g = wg[p];
        if (!(fabs(f) < kDwMax && fabs(g) < kDwMax)) flag |= 2;
        const int32_t id = A.vid[p];
        if (id != v) sum(id, f, g);  // padding names v itself
        wf48[p] = f;
        wg48[p] = g;
    }
    for (int64_t q = eb + (int64_t)kSell * sub; q < ee; q += kSell * kFoldLanes) {
        const double w = we[q];
        const float h = __double2float_rn(w);
        we48[q] = make_float2(h, __double2float_rn(w - (double)h));
        if (!(fabs(w) < kDwMax)) flag |= 2;
        edges += w != 0.0;
    }
    if (real && sub == kFoldLanes - 1) {
        double f = cfg[v], g = cfg[A.n_real + v];
        sum(v, f, g);
        cfg48[v] = f;
        cfg48[A.n_real + v] = g;
    }
    // every edge belongs to one entry or to the centre
    int miss = edges - found;
    for (int o = 1; o < kFoldLanes; o <<= 1) miss += __shfl_xor_sync(0xffffffffu, miss, o);
    if (real && miss != 0) flag |= 1;
    if (flag) atomicOr(bad, flag);
}
template <int MODE>
__global__ void __launch_bounds__(kDivBlock) div_f32_kernel(DivArgs A) {
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= A.n_real) return;
    if (MODE != 0 && A.dt_dev && *A.dt_dev == 0.0) return;  // adaptive run already at t_end
    div_f32_body<MODE>(A, v);
}

// Grid-wide barrier for a cooperative launch, with a bounded wait: thread 0
// of each block arrives on *count; the last arrival resets it and advances
// *gen; the others spin on *gen at most `limit` times (with a short sleep).
// Returns false (and sets *err) if the wait ran out.  Once *err is set no
// block arrives any more (a block finding it set at entry, or while it
// waits, gives up), so a count left short by a timed-out barrier is never
// completed by a later barrier of the same call; the host resets count,
// gen and err before the next call.
__device__ bool grid_barrier(unsigned int *count, volatile unsigned int *gen, unsigned int nblocks,
                             unsigned long long limit, int *err) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile int *verr = err;
        ok = 0;
        if (*verr == 0) {
            ok = 1;
            const unsigned int g = *gen;
            __threadfence();
            const unsigned int arrived = atomicAdd(count, 1u);
            if (arrived == nblocks - 1) {
                *count = 0;
                __threadfence();
                atomicAdd((unsigned int *)gen, 1u);
            } else {
                unsigned long long it = 0;
                while (*gen == g) {
                    if (*verr != 0 || ++it > limit) {
                        ok = 0;
                        atomicExch(err, 1);
                        break;
                    }
                    __nanosleep(64);
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// A persistent launch after a timed-out barrier of the same call does no
// work: its state would rest on a stage that did not complete.  Thread 0
// reads the flag for its block, so the whole block takes the same branch.
__device__ __forceinline__ bool barrier_failed(const int *err) {
    __shared__ int failed;
    if (threadIdx.x == 0) failed = *(const volatile int *)err;
    __syncthreads();
    return failed != 0;
}

// One SSP-RK3 stage over every mesh of a batch in one cooperative launch:
// all edge fluxes, a grid barrier, then every vertex's divergence and stage
// update (grid-stride loops; MODE = stage 1..3).  TILES (FP32): each kTile
// threads of a block take divergence tiles of their own, with T.smem bytes of
// the dynamic shared memory and a named barrier (1 .. blockDim / kTile).
template <int PREC, int MODE, bool TILES>
__global__ void stage_persistent_kernel(const __grid_constant__ EdgeArgs EA, const __grid_constant__ DivArgs DA,
                                        unsigned int *bar_count, unsigned int *bar_gen, unsigned int nblocks_expected,
                                        unsigned long long spin_limit, int *err,
                                        const __grid_constant__ TileTables T) {
    if (barrier_failed(err)) return;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t e = t0; e < EA.ne; e += stride) {
        if (PREC == 64) edge_flux_f64_body(EA, e);
        else if (EA.coef_gaps) edge_flux_f32_body<true>(EA, e);
        else edge_flux_f32_body<false>(EA, e);
    }
    __threadfence();
    if (!grid_barrier(bar_count, bar_gen, nblocks_expected, spin_limit, err)) return;
    if (TILES) {
        extern __shared__ float4 tile_stage[];
        const int group = (int)threadIdx.x / kTile, groups = (int)blockDim.x / kTile;
        float4 *sm = tile_stage + (int64_t)group * (T.smem / (int)sizeof(float4));
        // barrier numbers as constants: a register operand would reserve all 16 of
        // a block, and the SM's 64 then hold four blocks
        const auto sync = [group] {
            switch (group) {
                case 0: asm volatile("bar.sync 1, %0;" ::"n"(kTile) : "memory"); break;
                case 1: asm volatile("bar.sync 2, %0;" ::"n"(kTile) : "memory"); break;
                case 2: asm volatile("bar.sync 3, %0;" ::"n"(kTile) : "memory"); break;
                default: asm volatile("bar.sync 4, %0;" ::"n"(kTile) : "memory"); break;
            }
        };
        for (int64_t t = (int64_t)blockIdx.x * groups + group; t < T.ntiles; t += (int64_t)gridDim.x * groups) {
            div_f32_tile_body<MODE>(DA, T, t, (int)threadIdx.x % kTile, sm, sync);
            sync();  // the next tile's staging takes the same memory
        }
        return;
    }
    for (int64_t v = t0; v < DA.n_real; v += stride) {
        if (PREC == 64) div_f64_body<MODE>(DA, v);
        else div_f32_body<MODE>(DA, v);
    }
}

// Precision 48, and with GUARD precision 64: the same stage with the double-word edge flux (its staging in
// dynamic shared memory, kDwSlots 16-byte slots per thread) and the folded
// divergence.  At most 512 threads a block, so at most 128 registers.
template <int MODE, bool GUARD>
__global__ void __launch_bounds__(512, 1)
    stage_persistent_dw_kernel(const __grid_constant__ EdgeArgs EA, const __grid_constant__ DivArgs DA,
                               unsigned int *bar_count, unsigned int *bar_gen, unsigned int nblocks_expected,
                               unsigned long long spin_limit, int *err) {
    if (barrier_failed(err)) return;
    extern __shared__ float4 dw_stage[];
    const dwa::Stage T{dw_stage + threadIdx.x, (int)blockDim.x};
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const Wide wide = GUARD ? wide_batch_stage(EA) : kNone;
    for (int64_t c = t0; c <= EA.n_comp; c += stride) dwa::clear_wide(EA, c);
    for (int64_t e = t0; e < EA.ne; e += stride) {
        if (GUARD) edge_flux_guard_body(EA, e, T, wide);
        else dwa::edge_flux_dw_body<false>(EA, e, T);
    }
    __threadfence();
    if (!grid_barrier(bar_count, bar_gen, nblocks_expected, spin_limit, err)) return;
    for (int64_t v = t0; v < DA.n_real; v += stride) div_f64_any<MODE, GUARD ? kDivGuard : kDivDw>(DA, v, wide);
}

// ------------------------------------------------------------------ support kernels
// Smallest row index whose state has rho <= 0 (or NaN) or a non-finite
// momentum or energy (set_state's physical check).
__global__ void check_rows_kernel(const double *__restrict__ w, int64_t n, unsigned long long *bad) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const dbl4 s = ld4(w, i);
    if (!(s.x > 0.0) || !isfinite(s.y) || !isfinite(s.z) || !isfinite(s.w)) atomicMin(bad, (unsigned long long)i);
}

// zero (optional): words set to 0 on the way, which saves a memset's launch
// when a state is set (in a small mesh's 25 us residual call within the spread of
// the runs).
__global__ void permute_rows_kernel(const double *__restrict__ in, double *__restrict__ out,
                                    const int32_t *__restrict__ map, int64_t n, bool gather, double *zero, int nzero) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (zero && i < nzero) zero[i] = 0.0;
    if (i >= n) return;
    const int64_t m = __ldg(map + i);
    if (gather) st4(out, i, ld4(in, m));  // out[i] = in[map[i]]
    else st4(out, m, ld4(in, i));         // out[map[i]] = in[i]
}

// Ghost vertices (internal ids n_real .. n_real+n_ghost-1).  A transmissive
// ghost copies its donor's state and fluxes (reading of the configs'
// transmissive boundary); a Dirichlet ghost (its own donor) takes its fixed
// state and fluxes from wsrc / Fsrc, the buffers of the step's start state
// (a no-op when they are the buffers being filled).  F holds `fq` 16-byte
// words per vertex.
// (F, Fsrc) and (Q, Qsrc): vertex fluxes and, for an FP64 state, Roe records
// (2 words per vertex), in the one launch.
__global__ void ghost_fill_kernel(double *__restrict__ w, const double *wsrc, uint4 *__restrict__ F, const uint4 *Fsrc,
                                  int fq, uint4 *__restrict__ Q, const uint4 *Qsrc, float4 *__restrict__ w32,
                                  const int32_t *__restrict__ donor, int64_t n_real, int64_t n_ghost) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_ghost) return;
    const int64_t g = n_real + i, d = __ldg(donor + i);
    if (d == g) {
        if (w && wsrc && w != wsrc) st4(w, g, ld4(wsrc, g));
        if (F && Fsrc && F != Fsrc)
            for (int c = 0; c < fq; ++c) F[fq * g + c] = Fsrc[fq * g + c];
        if (Q && Qsrc && Q != Qsrc)
            for (int c = 0; c < 2; ++c) Q[2 * g + c] = Qsrc[2 * g + c];
        return;
    }
    if (w) st4(w, g, ld4(w, d));
    if (F)
        for (int c = 0; c < fq; ++c) F[fq * g + c] = F[fq * d + c];
    if (Q)
        for (int c = 0; c < 2; ++c) Q[2 * g + c] = Q[2 * d + c];
    if (w32) w32[g] = w32[d];
}

// h / (|u| + c) of a state (0 where it is non-physical)
__device__ __forceinline__ double dt_bound64(const dbl4 &s, double h, double gamma) {
    const double ir = 1.0 / s.x;
    const double u = s.y * ir, v = s.z * ir;
    const double p = (gamma - 1.0) * (s.w - 0.5 * (s.y * u + s.z * v));
    const double c = sqrt(gamma * p * ir);
    const double t = h / (sqrt(u * u + v * v) + c);
    return t > 0 ? t : 0.0;
}
// Adaptive step from the reduced bound in *slot; runs in one thread once every
// vertex has been reduced.  tstate = (t, dt, nonphysical); the slot is reset.
__device__ __forceinline__ void dt_finalize(unsigned long long *slot, double *tstate, double cfl, double t_end,
                                            unsigned long long *nsteps) {
    const double bound = __longlong_as_double((long long)*(volatile unsigned long long *)slot);
    const double t = tstate[0];
    double dt = cfl * bound;
    const double rem = t_end - t;
    if (!(bound > 0.0) || !(bound < INFINITY)) {
        dt = 0.0;
        tstate[2] = 1.0;  // non-physical state
    } else if (rem <= 1e-12 * fabs(t_end)) {
        dt = 0.0;
    } else if (rem < dt) {
        dt = rem;
    }
    tstate[1] = dt;
    tstate[0] = dt > 0.0 ? (rem < cfl * bound ? t_end : t + dt) : t;
    if (dt > 0.0) *nsteps += 1;
    *slot = 0x7FF0000000000000ull;
}
// min over vertices of h_v / (|u| + c), as the bit pattern of a positive double.
// The FP64 divisions and square roots (about 65 instructions of 64 cycles a
// warp) are taken only where the minimum can lie: the bound is estimated in
// FP32, and a vertex whose estimate is above the block's smallest, or above the
// minimum reduced so far, by more than 2^-10 is left out.  The estimate errs by
// a few 2^-24 relative, times the Mach number through the pressure; a vertex
// with p < 2^-10 rho E (Mach above 40), or outside FP32's comfortable range, is
// always taken, so the result is the FP64 minimum itself.  With `fin` (adaptive stepping) the last block
// also finalises the step.  1,000,000 vertices: 19.6 us (89 with every vertex
// in FP64 and the finalisation as a launch of its own); the state alone is 32
// MB.
constexpr int kDtBlock = 256;
__global__ void __launch_bounds__(kDtBlock)
    max_dt_kernel(const double *__restrict__ w, const double *__restrict__ hmin, int64_t n, double gamma,
                  unsigned long long *slot, const int32_t *__restrict__ comp, DtFinal fin) {
    __shared__ float smallest[kDtBlock / 32];
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool on = v < n;
    dbl4 s = dbl4_make(0, 0, 0, 0);
    double h = 0.0;
    float est = INFINITY;
    bool sure = false;
    if (on) {
        s = ld4(w, v);
        h = hmin[v];
        const float g = (float)gamma, r = (float)s.x, mx = (float)s.y, my = (float)s.z, E = (float)s.w;
        const float ir = 1.0f / r, ux = mx * ir, uy = my * ir;
        const float p = (g - 1.0f) * (E - 0.5f * (mx * ux + my * uy));
        const float speed = sqrtf(ux * ux + uy * uy) + sqrtf(g * p * ir);
        est = (float)h / speed;
        sure = !(p > 0x1p-10f * E && E > 0x1p-100f && speed > 0x1p-60f) || !(est > 0x1p-100f && est < INFINITY);
    }
    float m = sure ? INFINITY : est;
    for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) smallest[threadIdx.x / 32] = m;
    __syncthreads();
    for (int i = 0; i < kDtBlock / 32; ++i) m = fminf(m, smallest[i]);
    bool take = on && (sure || est <= m * (1.0f + 0x1p-10f));
    if (comp) {  // one slot per component
        // the block's smallest may belong to another component: compare with the component's own slot only
        unsigned long long *own = slot + (on ? __ldg(comp + v) : 0);
        const double so_far = __longlong_as_double((long long)__ldcg(own));
        take = on && (sure || (double)est <= so_far * (1.0 + 0x1p-10));
        if (take) atomicMin(own, (unsigned long long)__double_as_longlong(dt_bound64(s, h, gamma)));
        return;
    }
    if (take && !sure) {
        const double so_far = __longlong_as_double((long long)__ldcg(slot));
        take = (double)est <= so_far * (1.0 + 0x1p-10);
    }
    double t = INFINITY;
    if (take) t = dt_bound64(s, h, gamma);
    if (__any_sync(0xffffffffu, take)) {
        for (int o = 16; o > 0; o >>= 1) t = fmin(t, __shfl_xor_sync(0xffffffffu, t, o));
        if ((threadIdx.x & 31) == 0) atomicMin(slot, (unsigned long long)__double_as_longlong(t));
    }
    if (!fin.tstate) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(fin.done, 1u) == gridDim.x - 1) {
        *fin.done = 0;
        __threadfence();
        dt_finalize(slot, fin.tstate, fin.cfl, fin.t_end, fin.nsteps);
    }
}

// FMA-throughput probe: 8 independent chains x = x*a + b per thread.
template <class T>
__global__ void fma_probe_kernel(T *out, int iters, T a, T b) {
    T x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = (T)(threadIdx.x + k);
    for (int i = 0; i < iters; ++i) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = x[k] * a + b;
    }
    T s = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += x[k];
    out[(int64_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

// which: 0 recip64, 1 rsqrt64, 2 half64, 3 twice64
__global__ void recip_check_kernel(const double *x, double *y, int64_t n, int which) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = x[i];
    y[i] = which == 0 ? recip64(v) : which == 1 ? rsqrt64(v) : which == 2 ? half64(v) : twice64(v);
}

// the FP32 edge kernel's coefficient block of n edges from their gaps
__global__ void weno_coef32_check_kernel(const float4 *g, float *k, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float c[kCoefN];
    weno_coef32(g[i], c);
#pragma unroll
    for (int j = 0; j < kCoefN; ++j) k[(int64_t)kCoefN * i + j] = c[j];
}

inline unsigned blocks(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

}  // namespace

void launch_vertex_flux_f64(const double *w, double *F, int64_t n, double gamma, cudaStream_t s, double *Q, int *wide,
                            int64_t n_real, const int32_t *wcomp) {
    if (n > 0) vertex_flux_f64_kernel<<<blocks(n, 256), 256, 0, s>>>(w, F, Q, n, gamma - 1.0, wide, n_real, wcomp);
}
void launch_fold_tables(const DivArgs &a, const int32_t *left, const double *nx, const double *ny, double *wf48,
                        double *wg48, float2 *we48, double *cfg48, int *bad, cudaStream_t s) {
    if (a.n_real <= 0) return;
    const int64_t n = (a.n_real + kSell - 1) / kSell * kSell * kFoldLanes;
    fold_tables_kernel<<<blocks(n, 128), 128, 0, s>>>(a, left, nx, ny, wf48, wg48, we48, cfg48, bad);
}
void launch_vertex_flux_f32(const double *w, float4 *F, float4 *w32, int64_t n, double gamma, cudaStream_t s) {
    if (n > 0) vertex_flux_f32_kernel<<<blocks(n, 256), 256, 0, s>>>(w, F, w32, n, (float)(gamma - 1.0));
}
void launch_edge_flux_f64(const EdgeArgs &a, cudaStream_t s) {
    if (a.ne > 0) edge_flux_f64_kernel<<<blocks(a.ne, kEdgeBlock), kEdgeBlock, 0, s>>>(a);
}
void launch_edge_flux_guard(const EdgeArgs &a, cudaStream_t s) {
    if (a.ne > 0) edge_flux_guard_kernel<<<blocks(a.ne, kEdgeBlock), kEdgeBlock, 0, s>>>(a);
}
void launch_edge_flux_f32(const EdgeArgs &a, cudaStream_t s) {
    if (a.ne <= 0) return;
    if (a.coef_gaps) edge_flux_f32_kernel<true><<<blocks(a.ne, kEdgeBlock), kEdgeBlock, 0, s>>>(a);
    else edge_flux_f32_kernel<false><<<blocks(a.ne, kEdgeBlock), kEdgeBlock, 0, s>>>(a);
}
template <int KIND, int LPV>
void launch_div_f64_t(const DivArgs &a, int mode, cudaStream_t s) {
    const unsigned g = blocks(a.n_real * LPV, kDivBlock);
    switch (mode) {
        case 0: div_f64_kernel<0, KIND, LPV><<<g, kDivBlock, 0, s>>>(a); break;
        case 1: div_f64_kernel<1, KIND, LPV><<<g, kDivBlock, 0, s>>>(a); break;
        case 2: div_f64_kernel<2, KIND, LPV><<<g, kDivBlock, 0, s>>>(a); break;
        default: div_f64_kernel<3, KIND, LPV><<<g, kDivBlock, 0, s>>>(a); break;
    }
}
template <int LPV>
void launch_div_f64_l(const DivArgs &a, int mode, cudaStream_t s) {
    if (a.kind == kDivGuard) launch_div_f64_t<kDivGuard, LPV>(a, mode, s);
    else if (a.kind == kDivDw) launch_div_f64_t<kDivDw, LPV>(a, mode, s);
    else launch_div_f64_t<kDivPlain, LPV>(a, mode, s);
}
void launch_div_f64(const DivArgs &a, int mode, cudaStream_t s) {
    if (a.n_real <= 0) return;
    // Small meshes leave most of the chip's 152 x 24 resident warps empty while
    // each thread walks 60 to 100 dependent gathers, so several lanes share a
    // vertex.  RK3 step of the vortex at 1, 2, 4 lanes: 4096 vertices 84 / 68 / 56
    // us, 10,000 94 / 82 / 79, 16,900 107 / 98 / 101, 48,400 195 / 183 / 214, 67,600
    // 241 / 255 / 289 (the stage update is repeated by every warp, so more lanes
    // cost FP64 time once the warps are there); 8 lanes win only below 2000.
    if (a.n_real <= 12 * 1024) launch_div_f64_l<4>(a, mode, s);
    else if (a.n_real <= 56 * 1024) launch_div_f64_l<2>(a, mode, s);
    else launch_div_f64_l<1>(a, mode, s);
}
void launch_div_f32(const DivArgs &a, int mode, cudaStream_t s) {
    if (a.n_real <= 0) return;
    const unsigned g = blocks(a.n_real, kDivBlock);
    switch (mode) {
        case 0: div_f32_kernel<0><<<g, kDivBlock, 0, s>>>(a); break;
        case 1: div_f32_kernel<1><<<g, kDivBlock, 0, s>>>(a); break;
        case 2: div_f32_kernel<2><<<g, kDivBlock, 0, s>>>(a); break;
        default: div_f32_kernel<3><<<g, kDivBlock, 0, s>>>(a); break;
    }
}
void launch_tile_count(const TileSource &S, const TileTables &T, int32_t *nv, int32_t *ne, int32_t *gv, int32_t *ge,
                       cudaStream_t s) {
    if (T.ntiles > 0)
        tile_count_kernel<<<dim3((unsigned)T.ntiles, 2), kTileThreads, sizeof(TileWork), s>>>(S, T, nv, ne, gv, ge);
}
void launch_tile_fill(const TileSource &S, const TileTables &T, cudaStream_t s) {
    if (T.ntiles > 0) tile_fill_kernel<<<dim3((unsigned)T.ntiles, 2), kTileThreads, sizeof(TileWork), s>>>(S, T);
}
void launch_div_f32_tiles(const DivArgs &a, const TileTables &t, int mode, cudaStream_t s) {
    const unsigned g = (unsigned)t.ntiles;
    switch (mode) {
        case 0: div_f32_tile_kernel<0><<<g, kTile, t.smem, s>>>(a, t); break;
        case 1: div_f32_tile_kernel<1><<<g, kTile, t.smem, s>>>(a, t); break;
        case 2: div_f32_tile_kernel<2><<<g, kTile, t.smem, s>>>(a, t); break;
        default: div_f32_tile_kernel<3><<<g, kTile, t.smem, s>>>(a, t); break;
    }
}
void launch_check_rows(const double *w, int64_t n, unsigned long long *bad, cudaStream_t s) {
    if (n > 0) check_rows_kernel<<<blocks(n, 256), 256, 0, s>>>(w, n, bad);
}
void launch_permute_rows(const double *in, double *out, const int32_t *map, int64_t n, bool gather, cudaStream_t s,
                         double *zero, int nzero) {
    if (n > 0) permute_rows_kernel<<<blocks(n, 256), 256, 0, s>>>(in, out, map, n, gather, zero, nzero);
}
void launch_ghost_fill(double *w, const double *wsrc, void *F, const void *Fsrc, int fq, double *Q, const double *Qsrc,
                       float4 *w32, const int32_t *donor, int64_t n_real, int64_t n_ghost, cudaStream_t s) {
    if (n_ghost > 0)
        ghost_fill_kernel<<<blocks(n_ghost, 256), 256, 0, s>>>(
            w, wsrc, static_cast<uint4 *>(F), static_cast<const uint4 *>(Fsrc), fq, reinterpret_cast<uint4 *>(Q),
            reinterpret_cast<const uint4 *>(Qsrc), w32, donor, n_real, n_ghost);
}
void launch_max_dt(const double *w, const double *hmin, int64_t n, double gamma, unsigned long long *slot,
                   cudaStream_t s, const int32_t *comp, const DtFinal &fin) {
    if (n > 0 || fin.tstate) max_dt_kernel<<<blocks(n > 0 ? n : 1, kDtBlock), kDtBlock, 0, s>>>(w, hmin, n, gamma, slot, comp, fin);
}

namespace {
// Dynamic shared memory of the FP32 persistent stage, 0 where it does without
// tiles: kTileGroups groups of kTile threads have to fit an SM, as many as the
// kernel's registers allow, so that every launch shape that fits without the
// staging fits with it.
constexpr int kTileGroups = 6;
size_t persistent_tile_bytes(const TileTables &t, int threads) {
    const size_t bytes = (size_t)t.smem * (threads / kTile);
    return t.smem > 0 && (size_t)t.smem * kTileGroups <= (size_t)220 * 1024 ? bytes : 0;
}
template <int PREC, int MODE, bool TILES>
cudaError_t coop_t(const EdgeArgs &ea, const DivArgs &da, unsigned int *c, unsigned int *g, unsigned int ne,
                   unsigned long long lim, int *err, int threads, int nb, const TileTables &tt, size_t bytes,
                   cudaStream_t s) {
    EdgeArgs a = ea;
    DivArgs d = da;
    TileTables t = tt;
    void *args[] = {&a, &d, &c, &g, &ne, &lim, &err, &t};
    const void *k = (const void *)stage_persistent_kernel<PREC, MODE, TILES>;
    if (bytes > 0) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
    }
    return cudaLaunchCooperativeKernel(k, dim3(nb), dim3(threads), args, bytes, s);
}
template <int PREC, int MODE>
cudaError_t coop(const EdgeArgs &ea, const DivArgs &da, unsigned int *c, unsigned int *g, unsigned int ne,
                 unsigned long long lim, int *err, int threads, int nb, const TileTables &t, cudaStream_t s) {
    const size_t bytes = PREC == 32 ? persistent_tile_bytes(t, threads) : 0;
    if (bytes > 0) return coop_t<PREC, MODE, PREC == 32>(ea, da, c, g, ne, lim, err, threads, nb, t, bytes, s);
    return coop_t<PREC, MODE, false>(ea, da, c, g, ne, lim, err, threads, nb, t, 0, s);
}
}  // namespace

namespace {
size_t dw_stage_bytes(int threads) { return (size_t)dwa::kDwSlots * sizeof(float4) * threads; }
template <int MODE, bool GUARD>
cudaError_t coop48(const EdgeArgs &ea, const DivArgs &da, unsigned int *c, unsigned int *g, unsigned int ne,
                   unsigned long long lim, int *err, int threads, int nb, cudaStream_t s) {
    EdgeArgs a = ea;
    DivArgs d = da;
    void *args[] = {&a, &d, &c, &g, &ne, &lim, &err};
    const size_t bytes = dw_stage_bytes(threads);
    cudaError_t e = cudaFuncSetAttribute((const void *)stage_persistent_dw_kernel<MODE, GUARD>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return e;
    return cudaLaunchCooperativeKernel((const void *)stage_persistent_dw_kernel<MODE, GUARD>, dim3(nb), dim3(threads), args,
                                       bytes, s);
}
}  // namespace

cudaError_t launch_stage_persistent(int prec, int mode, const EdgeArgs &ea, const DivArgs &da, unsigned int *bar_count,
                                    unsigned int *bar_gen, unsigned int nblocks_expected,
                                    unsigned long long spin_limit, int *err, int threads, int nb, const TileTables &t,
                                    cudaStream_t s) {
    const unsigned int ne = nblocks_expected;
    if (prec == 48) {
        if (mode == 1) return coop48<1, false>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, s);
        if (mode == 2) return coop48<2, false>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, s);
        return coop48<3, false>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, s);
    }
    if (prec == 64 && da.kind == kDivGuard) {
        if (mode == 1) return coop48<1, true>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, s);
        if (mode == 2) return coop48<2, true>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, s);
        return coop48<3, true>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, s);
    }
    if (prec == 64) {
        if (mode == 1) return coop<64, 1>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, t, s);
        if (mode == 2) return coop<64, 2>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, t, s);
        return coop<64, 3>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, t, s);
    }
    if (mode == 1) return coop<32, 1>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, t, s);
    if (mode == 2) return coop<32, 2>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, t, s);
    return coop<32, 3>(ea, da, bar_count, bar_gen, ne, spin_limit, err, threads, nb, t, s);
}

namespace {
template <bool GUARD>
int dw_blocks_per_sm(int threads) {
    int n = 0;
    const size_t bytes = dw_stage_bytes(threads);
    for (auto k : {stage_persistent_dw_kernel<1, GUARD>, stage_persistent_dw_kernel<2, GUARD>,
                   stage_persistent_dw_kernel<3, GUARD>})
        if (cudaFuncSetAttribute((const void *)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess)
            return 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, stage_persistent_dw_kernel<3, GUARD>, threads, bytes);
    return n;
}
}  // namespace

int persistent_blocks_per_sm(int prec, int threads, bool guard, const TileTables &t) {
    int n = 0;
    // the three stage modes share their register footprint; mode 3 stands for all
    if (prec == 48) return dw_blocks_per_sm<false>(threads);
    if (prec == 64) {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, stage_persistent_kernel<64, 3, false>, threads, 0);
        // a block the FP64 kernel has no registers for is refused at precision 64 on either path
        return guard && n > 0 ? dw_blocks_per_sm<true>(threads) : n;
    }
    const size_t bytes = persistent_tile_bytes(t, threads);
    if (bytes > 0) {
        for (auto k : {stage_persistent_kernel<32, 1, true>, stage_persistent_kernel<32, 2, true>,
                       stage_persistent_kernel<32, 3, true>})
            if (cudaFuncSetAttribute((const void *)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) !=
                cudaSuccess)
                return 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, stage_persistent_kernel<32, 3, true>, threads, bytes);
    } else {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, stage_persistent_kernel<32, 3, false>, threads, 0);
    }
    return n;
}

double fma_probe_tflops(int precision, int sms, void *scratch, cudaStream_t s) {
    const int nb = sms * 8, nt = 256;
    const int iters = precision == 64 ? 2048 : 65536;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    for (int rep = 0; rep < 2; ++rep) {  // first launch warms up
        cudaEventRecord(a, s);
        if (precision == 64)
            fma_probe_kernel<double><<<nb, nt, 0, s>>>(static_cast<double *>(scratch), iters, 0.999999, 1e-7);
        else
            fma_probe_kernel<float><<<nb, nt, 0, s>>>(static_cast<float *>(scratch), iters, 0.999999f, 1e-7f);
        cudaEventRecord(b, s);
    }
    cudaEventSynchronize(b);
    float ms = 0;
    cudaEventElapsedTime(&ms, a, b);
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    return 2.0 * 8.0 * iters * (double)nb * nt / (ms * 1e-3) / 1e12;
}

void launch_recip_check(const double *x, double *y, int64_t n, int which, cudaStream_t s) {
    if (n > 0) recip_check_kernel<<<blocks(n, 256), 256, 0, s>>>(x, y, n, which);
}

void launch_weno_coef32_check(const float4 *g, float *k, int64_t n, cudaStream_t s) {
    if (n > 0) weno_coef32_check_kernel<<<blocks(n, 256), 256, 0, s>>>(g, k, n);
}

}  // namespace fdu
