// Extended source indices of the periodic box (range.cu, range_fp32.cu): e in [-M, 2M) is spring e mod M
// shifted by 2 pi floor(e / M); in free space e lies in [0, M).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "internal.h"

namespace wave1d {

constexpr double kPiR = 3.14159265358979323846264338327950288;

// position of extended source index e: the same expression as the host's window tests
__device__ __forceinline__ double rs_xext(const DevPlan& P, int64_t e) {
    if (e < 0) return P.x[e + P.M] - 2.0 * kPiR;
    if (e >= P.M) return P.x[e - P.M] + 2.0 * kPiR;
    return P.x[e];
}

__device__ __forceinline__ int64_t rs_spring(int64_t e, int64_t M) { return e < 0 ? e + M : (e >= M ? e - M : e); }

}  // namespace wave1d
