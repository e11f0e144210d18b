// What the double-word edge flux (fdu_dw_edge.cuh) and its adjoint share
// besides the arithmetic (device only): the order of the paired coefficient
// block, 4-vectors and FP64 loads.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "fdu_dw.cuh"
#include "fdu_internal.h"

namespace fdu {
namespace dwa {

// Values (of the kEdgeCoef block) in lane 0 and 1 of pair p of the paired block.
__device__ constexpr int dw_pair(int p, int lane) {
    constexpr int t[kDwPairs][2] = {{0, 15}, {1, 16}, {2, 17}, {3, 18}, {4, 19},   {5, 11},  {6, 10},
                                    {7, 14}, {8, 13}, {9, 12}, {20, 22}, {21, 23}, {kCoefN, kCoefN + 1}};
    return t[p][lane];
}

struct dw4 {
    dw x, y, z, w;
};
__device__ __forceinline__ dw4 d4(dw x, dw y, dw z, dw w) { return dw4{x, y, z, w}; }
struct d4v {
    double x, y, z, w;
};
__device__ __forceinline__ d4v ldd4(const double *p, int64_t i) {
    const double2 a = __ldg(reinterpret_cast<const double2 *>(p) + 2 * i);
    const double2 b = __ldg(reinterpret_cast<const double2 *>(p) + 2 * i + 1);
    return d4v{a.x, a.y, b.x, b.y};
}

template <bool BOUNDED = false>
__device__ __forceinline__ dw4 d2dw4(const d4v &v) {
    return d4(d2dw<BOUNDED>(v.x), d2dw<BOUNDED>(v.y), d2dw<BOUNDED>(v.z), d2dw<BOUNDED>(v.w));
}

}  // namespace dwa
}  // namespace fdu
