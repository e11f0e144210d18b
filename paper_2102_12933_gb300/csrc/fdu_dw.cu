// Edge flux with FP64-level accuracy in double-word FP32 arithmetic.
//
// The same function as edge_flux_f64 (Section 2.3.1 and the Appendix:
// characteristic NU-WENO5 from both sides, Roe flux with Harten's entropy
// fix), arranged so that everything of the size of the state runs in FP64
// and everything of the size of an increment runs in double words (FP32
// pairs, about 48 significant bits), which GB300 executes on its FP32
// pipes at 64 times the FP64 instruction rate.
//
//   FP64 : the five stencil differences R1-L1, L2-L1, L3-L1, R2-R1, R3-R1
//          (exact or correctly rounded); the normal flux F_n(L1) of the
//          edge's left vertex, which the divergence adds through its folded
//          FP64 vertex weights (div_f64_body<MODE, true>).
//   DW   : characteristic projection at the Roe average of (L1, R1), the
//          WENO increments, the flux increment F_n(w_L) - F_n(L1) in a
//          cancellation-free form, and the Roe dissipation
//          D = R diag((lambda - |lambda|_fix)/2) L (w_R - w_L); the kernel
//          writes r - F_n(L1) = [F_n(w_L) - F_n(L1)] + D as double words.
// An error of relative size 2^-46 in an increment of size h |grad w| gives
// an error of that size times h in the flux, which the least-squares
// divergence (weights of size 1/h) does not amplify beyond the FP64 path's
// own rounding.  The NU-WENO5 and edge-flux bodies are in fdu_dw_edge.cuh
// (shared with the batched persistent stage).
//
// FP32 has a narrower exponent range than FP64.  The smoothness indicators
// are formed from the differences of each field scaled by a power of two
// (max |difference| in [1/2, 1)), with epsilon scaled by its square, so the
// nonlinear weights (invariant under a common scale of beta + epsilon) are
// unchanged; beta + epsilon is bounded below by 2^-100, which moves only
// weights between sub-stencils whose differences are below 2^-50 of the
// field's largest, whose values then differ by less than that.  The weights
// are formed as alpha_k = C_k / (beta_k + eps), omega = alpha / sum(alpha):
// the same quotient as the FP64 kernel's product form.
//
// What bounds it: the FMA pipe (67 % busy) and the issue slots and instruction
// fetch in front of it.  The left and right states (and the projections of the
// mirrored differences) run in the two lanes of packed FP32 instructions, in
// the edge's own frame, with sums and products that leave their low words
// unnormalised where no product of two of them follows: about 4200 FP32
// operations per edge in half the issue slots, against 5250 one to a slot.
// 128 registers, 16 warps per SM.  0.1742 -> 0.116 ms at 250k vertices (750k
// edges); the FMA pipe alone would take 0.079 ms.
#include <cuda_runtime.h>

#include <cstdint>

#include "fdu_dw.cuh"
#include "fdu_dw_euler.cuh"
#include "fdu_dw_edge.cuh"
#include "fdu_internal.h"
#include "fdu_kernels.cuh"

namespace fdu {
namespace {

using namespace dwa;

__global__ void __launch_bounds__(kEdgeBlock, 4) edge_flux_dw_kernel(EdgeArgs A) {
    __shared__ float4 stage[kDwSlots * kEdgeBlock];
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= A.ne) return;
    if (A.dt_dev && *A.dt_dev == 0.0) return;
    clear_wide(A, e);
    edge_flux_dw_body<false>(A, e, Stage{stage + threadIdx.x, kEdgeBlock});
}

// The edge coefficient block as paired double words: hi = the FP32 rounding
// of a value, lo = the FP32 rounding of the remainder.
__global__ void coef_dw_kernel(const double *__restrict__ coef, float4 *__restrict__ out, int64_t ne,
                               int *bad) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= ne) return;
#pragma unroll
    for (int p = 0; p < kDwPairs; ++p) {
        const double a = coef[(int64_t)dw_pair(p, 0) * ne + e], b = coef[(int64_t)dw_pair(p, 1) * ne + e];
        if (!(fabs(a) < kDwMax && fabs(b) < kDwMax)) atomicOr(bad, 2);
        const float ah = __double2float_rn(a), bh = __double2float_rn(b);
        out[(int64_t)p * ne + e] = make_float4(ah, bh, __double2float_rn(a - (double)ah), __double2float_rn(b - (double)bh));
    }
}

// The normalised algorithms, for the accuracy check alone (operations 1 to 6), as
// analysed by Joldes, Muller and Popescu, "Tight and rigorous error bounds for
// basic building blocks of double-word arithmetic", ACM TOMS 44(2), 2017:
//   add      accurate sum (their Algorithm 6): relative error <= 3u^2
//   add_sl   sloppy sum (Algorithm 5): absolute error about u^2 (|x| + |y|)
//   mul      double-word product (Algorithm 11): relative error <= 5u^2
//   mul_u    the same before its final Fast2Sum, for operands of a sum
// with u = 2^-24.  The reciprocal and the reciprocal square root take the
// FP32 hardware approximation (PTX rcp.approx / rsqrt.approx, relative error
// below 2^-22) and one correction of second order in its residual e:
//   1/x       = r (1 + e + e^2 + ...),      e = 1 - x r
//   1/sqrt(x) = y (1 + e/2 + 3e^2/8 + ...), e = 1 - x y^2
// leaving O(e^3) < 2^-60 besides the double-word rounding.
// s + t = a + b exactly, for |a| >= |b| (or a = 0)
__device__ __forceinline__ dw fast_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return dw{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ dw add(dw x, dw y) {
    const dw s = two_sum(x.h, y.h);
    const dw t = two_sum(x.l, y.l);
    const dw v = fast_two_sum(s.h, __fadd_rn(s.l, t.h));
    return fast_two_sum(v.h, __fadd_rn(t.l, v.l));
}
__device__ __forceinline__ dw add_sl(dw x, dw y) {
    const dw s = two_sum(x.h, y.h);
    return fast_two_sum(s.h, __fadd_rn(s.l, __fadd_rn(x.l, y.l)));
}
__device__ __forceinline__ dw mul(dw x, dw y) {
    const float ch = __fmul_rn(x.h, y.h);
    const float cl1 = __fmaf_rn(x.h, y.h, -ch);
    const float cl2 = __fmaf_rn(x.l, y.h, __fmul_rn(x.h, y.l));
    return fast_two_sum(ch, __fadd_rn(cl1, cl2));
}
// The same product without the final renormalisation (|l| may reach about
// 2 ulp(h)): for operands of a sum, which renormalises.
__device__ __forceinline__ dw mul_u(dw x, dw y) {
    const float ch = __fmul_rn(x.h, y.h);
    const float cl1 = __fmaf_rn(x.h, y.h, -ch);
    return dw{ch, __fadd_rn(cl1, __fmaf_rn(x.l, y.h, __fmul_rn(x.h, y.l)))};
}
__device__ __forceinline__ dw recip(dw x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x.h));
    const float p = __fmul_rn(x.h, r);
    const float ep = __fmaf_rn(x.h, r, -p);  // x.h r = p + ep exactly; 1 - p is exact (p near 1)
    const float e = __fsub_rn(__fsub_rn(__fsub_rn(1.0f, p), ep), __fmul_rn(x.l, r));
    return fast_two_sum(r, __fmul_rn(r, __fmaf_rn(e, e, e)));
}
__device__ __forceinline__ dw rsqrt(dw x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x.h));
    const float y2 = __fmul_rn(y, y);
    const float y2l = __fmaf_rn(y, y, -y2);  // y^2 = y2 + y2l exactly
    const float p = __fmul_rn(x.h, y2);
    const float ep = __fmaf_rn(x.h, y2, -p);  // x.h y2 = p + ep exactly
    const float e = __fsub_rn(__fsub_rn(1.0f, p), __fadd_rn(ep, __fmaf_rn(x.h, y2l, __fmul_rn(x.l, y2))));
    return fast_two_sum(y, __fmul_rn(__fmul_rn(y, e), __fmaf_rn(0.375f, e, 0.5f)));
}

// The lean forms on one lane (float) or two (f2): operation k of a, b and c.
template <class T>
__device__ dwv<T> lean_op(int k, dwv<T> a, dwv<T> b, dwv<T> c) {
    switch (k) {
        case 0: return ladd(a, b);
        case 1: return lmul(a, b);
        case 2: return lfma(a, b, c);
        case 3: return lfma(ladd(a, c), b, c);  // an operand that is not normalised
        case 4: return lrecip(a);
        case 5: return lrsqrt(a);
        default: {
            const dwv<T> r = norm(ladd(a, b));
            return dwv<T>{r.h, fsub(r.h, r.h)};
        }
    }
}
// Accuracy check: inputs and outputs as doubles (inputs split by d2dw, outputs
// recombined exactly by dw2d).
__global__ void dw_check_kernel(int op, const double *__restrict__ x, const double *__restrict__ y,
                                double *__restrict__ z, int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    auto out = [&](dw r) { z[i] = dw2d(r); };
    if (op == 7) {  // compensated dot product of 8 consecutive pairs
        if (i >= n / 8) return;
        dot2 A{0.0f, 0.0f};
        for (int j = 0; j < 8; ++j) dot2_add(A, d2dw(x[8 * i + j]), d2dw(y[8 * i + j]));
        out(dot2_result(A));
        return;
    }
    if (i >= n) return;
    const dw a = d2dw(x[i]), b = d2dw(y[i]);
    if (op >= 8) {  // 8 + k alone; 16 + k and 24 + k in lane 0 and 1, the neighbour's operands in the other
        const int64_t j = i ^ 1;
        const dw a1 = d2dw(x[j]), b1 = d2dw(y[j]);
        if (op < 16) out(lean_op(op - 8, a, b, b1));
        else if (op < 24) out(first(lean_op(op - 16, pair(a, a1), pair(b, b1), pair(b1, b))));
        else out(second(lean_op(op - 24, pair(a1, a), pair(b1, b), pair(b, b1))));
        return;
    }
    switch (op) {
        case 0: out(a); break;
        case 1: out(add(a, b)); break;
        case 2: out(add_sl(a, b)); break;
        case 3: out(mul(a, b)); break;
        case 4: out(mul_u(a, b)); break;
        case 5: out(recip(a)); break;
        default: out(rsqrt(a)); break;
    }
}

}  // namespace

void launch_dw_check(int op, const double *x, const double *y, double *z, int64_t n, cudaStream_t s) {
    if (n > 0) dw_check_kernel<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(op, x, y, z, n);
}

void launch_coef_dw(const double *coef, float4 *coefdw, int64_t ne, int *bad, cudaStream_t s) {
    if (ne > 0) coef_dw_kernel<<<(unsigned)((ne + 255) / 256), 256, 0, s>>>(coef, coefdw, ne, bad);
}

void launch_edge_flux_dw(const EdgeArgs &a, cudaStream_t s) {
    if (a.ne > 0) edge_flux_dw_kernel<<<(unsigned)((a.ne + kEdgeBlock - 1) / kEdgeBlock), kEdgeBlock, 0, s>>>(a);
}

}  // namespace fdu
