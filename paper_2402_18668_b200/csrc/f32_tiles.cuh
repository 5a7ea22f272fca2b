// Register-tiled fp32 products on shared-memory tiles of 64 tokens (256 threads), and the symmetric feature rows
// psi(x) that they contract.  Both operands of a product lie row by row along the summation index: a float4 holds two
// operand pairs of the two-wide FMA, even and odd terms are summed apart.  Row pitches are chosen so that the float4s
// of eight consecutive rows fall into eight different bank groups (156, 68 and 20 floats).
// One operand of every product is the same for all 32 lanes and the other differs from lane to lane: a 128-bit
// shared-memory load of a warp takes two passes in the first case (measured) and four in the second.
#pragma once
#include "common.cuh"

namespace based {

constexpr int kFeat = 156;         // 153 symmetric features, zero padded to a multiple of 4
constexpr int kTF = 5;             // features per lane of a state tile
constexpr int kFeatRows = 160;     // = 32 kTF
constexpr int kRowT = 68;          // row pitch of tiles with 64 tokens per row
constexpr int kRowX = 20;          // row pitch of q / k tiles: 16 values, then 1 (0 past the end)
constexpr float kRsqrt2 = 0.70710678118654752f;

__device__ __forceinline__ void fma2(float2& acc, float ax, float ay, float bx, float by) {
    uint64_t r, a, b;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(acc.x), "f"(acc.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(ax), "f"(ay));
    asm("mov.b64 %0, {%1, %2};" : "=l"(b) : "f"(bx), "f"(by));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(r) : "l"(a), "l"(b));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(acc.x), "=f"(acc.y) : "l"(r));
}
__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// feature f = scale * x[m] * x[n] on a row whose element 16 is the constant 1
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

// up to 64 rows of 16 values -> [64][20]; rows past nt are zero, element 16 is 1 on real rows
__device__ __forceinline__ void load_x(float* dst, const float* __restrict__ src, int nt, int tid) {
    const int t = tid >> 2, p = tid & 3;
    const bool live = t < nt;
    *reinterpret_cast<float4*>(&dst[t * kRowX + 4 * p]) =
        live ? __ldg(reinterpret_cast<const float4*>(src + (size_t)t * kDFeat) + p) : make_float4(0.f, 0.f, 0.f, 0.f);
    if (p == 0) dst[t * kRowX + kDFeat] = live ? 1.f : 0.f;
}
// 64 tokens x up to 64 columns (a multiple of 4) of a row-major array, transposed -> [64 columns][68]
__device__ __forceinline__ void load_vt(float* dst, const float* __restrict__ src, int pitch, int ncol, int nt, int tid) {
    const int t = (tid & 7) + 8 * (tid >> 5);
    float4 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c4 = ((tid >> 3) & 3) + 4 * i;
        x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t < nt && 4 * c4 < ncol) x[i] = __ldg(reinterpret_cast<const float4*>(src + (size_t)t * pitch) + c4);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int c = 4 * (((tid >> 3) & 3) + 4 * i);
        dst[(c + 0) * kRowT + t] = x[i].x;
        dst[(c + 1) * kRowT + t] = x[i].y;
        dst[(c + 2) * kRowT + t] = x[i].z;
        dst[(c + 3) * kRowT + t] = x[i].w;
    }
}
// psi of the rows warp + 8 i of x, written by the warp that uses them: [64][156]
template <int NI>
__device__ __forceinline__ void psi_rows(float* dst, const float* x, const FeatTab& tab, int warp, int lane) {
#pragma unroll
    for (int i = 0; i < kTF; ++i) {
        const int f = lane + 32 * i;
        if (f >= kFeat) continue;
        const int m = tab.mn[f] & 255, n = tab.mn[f] >> 8;
        const float c = tab.scale[f];
#pragma unroll
        for (int u = 0; u < NI; ++u) {
            const int t = warp + 8 * u;
            dst[t * kFeat + f] = c * x[t * kRowX + m] * x[t * kRowX + n];
        }
    }
}
// psi transposed, tokens below nt rounded up to 4: [160][68]
__device__ __forceinline__ void psi_transposed(float* dst, const float* x, const FeatTab& tab, int nt, int tid) {
    const int lane = tid & 31, warp = tid >> 5;
    const int nq = (nt + 3) >> 2;                    // groups of four tokens
    for (int e = warp; e < kTF * nq; e += 8) {
        const int i = e / nq, t = (e - i * nq) * 4;
        const int f = lane + 32 * i;
        const int m = tab.mn[f] & 255, n = tab.mn[f] >> 8;
        const float c = tab.scale[f];
        float4 r;
        r.x = c * x[t * kRowX + m] * x[t * kRowX + n];
        r.y = c * x[(t + 1) * kRowX + m] * x[(t + 1) * kRowX + n];
        r.z = c * x[(t + 2) * kRowX + m] * x[(t + 2) * kRowX + n];
        r.w = c * x[(t + 3) * kRowX + m] * x[(t + 3) * kRowX + n];
        *reinterpret_cast<float4*>(&dst[f * kRowT + t]) = r;
    }
}
// acc[i][j] += sum_t psiT[lane + 32 i][t] vt[8 warp + j][t]
__device__ __forceinline__ void state_update(float2 (&acc)[kTF][8], const float* psi_t, const float* vt, int nt, int warp,
                                             int lane) {
    for (int t = 0; t < nt; t += 4) {
        float4 a[kTF];
#pragma unroll
        for (int i = 0; i < kTF; ++i) a[i] = lds4(&psi_t[(lane + 32 * i) * kRowT + t]);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float4 b = lds4(&vt[(warp * 8 + j) * kRowT + t]);
#pragma unroll
            for (int i = 0; i < kTF; ++i) fma2(acc[i][j], a[i].x, a[i].y, b.x, b.y);
#pragma unroll
            for (int i = 0; i < kTF; ++i) fma2(acc[i][j], a[i].z, a[i].w, b.z, b.w);
        }
    }
}
// sum over the tokens of one feature row
__device__ __forceinline__ float row_sum(const float* psi_t, int f, int nt) {
    float s0 = 0.f, s1 = 0.f;
    for (int t = 0; t < nt; t += 4) {
        const float4 a = lds4(&psi_t[f * kRowT + t]);
        s0 += a.x + a.y;
        s1 += a.z + a.w;
    }
    return s0 + s1;
}
// o[i][j] += sum_k a[warp + 8 i][k] b[lane + 32 j][k], k < nk (a multiple of 4)
template <int NI, int SA, int SB>
__device__ __forceinline__ void rows_product(float2 (&o)[NI][2], const float* a, const float* b, int nk, int warp, int lane) {
    const float* pa = a + warp * SA;
    const float* pb = b + lane * SB;
#pragma unroll 2
    for (int k = 0; k < nk; k += 4) {
        float4 y[2];
        y[0] = lds4(pb + k);
        y[1] = lds4(pb + 32 * SB + k);
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            const float4 x = lds4(pa + 8 * i * SA + k);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                fma2(o[i][j], x.x, x.y, y[j].x, y[j].y);
                fma2(o[i][j], x.z, x.w, y[j].z, y[j].w);
            }
        }
    }
}

}  // namespace based
