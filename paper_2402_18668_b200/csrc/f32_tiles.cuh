// What the fp32 kernels share: shared-memory loads and two-wide multiply-adds of register-tiled products whose operands
// lie along the summation index ([k][row], [k][column]), and the symmetric feature rows psi(x).
// A 128-bit shared-memory load of a warp takes two passes where neighbouring lanes 2n and 2n + 1 share an address (or all
// lanes do) and four otherwise (measured), so a thread's tile is 8 rows x 4 columns with lane bit 0 on the rows and the
// other bits on the columns: six passes per 32 multiply-adds.
#pragma once
#include "common.cuh"

namespace based {

constexpr float kRsqrt2 = 0.70710678118654752f;

__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }
// two products per instruction: acc += (x0, x1) * (y, y)
__device__ __forceinline__ void fma_pair(float2& acc, float x0, float x1, float y) {
    uint64_t r, a, b;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(acc.x), "f"(acc.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(x0), "f"(x1));
    asm("mov.b64 %0, {%1, %1};" : "=l"(b) : "f"(y));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(r) : "l"(a), "l"(b));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(acc.x), "=f"(acc.y) : "l"(r));
}

// psi: feature f = scale * x[m] * x[n] on a row whose element 16 is 1 (order of based_decode_step_sym, zero past the last)
constexpr int kFeat = 156;         // 153 features, padded to a multiple of 4
constexpr int kFeatRows = 160;     // padded to ten per thread of sixteen
struct FeatTab {
    uint32_t mn[kFeatRows];        // m | n << 8
    float scale[kFeatRows];
};
__device__ __forceinline__ void fill_feat_tab(FeatTab& t, int tid) {
    if (tid < kFeatRows) {
        int m = kDFeat, n = kDFeat;
        float c = 0.f;
        if (tid == 0) c = 1.f;
        else if (tid <= kDFeat) { m = tid - 1; c = kLinScale; }
        else if (tid < kDSym) { pair_of(tid - 1 - kDFeat, m, n); c = m == n ? kQuadScale : 0.25f; }
        t.mn[tid] = m | n << 8;
        t.scale[tid] = c;
    }
}

}  // namespace based
