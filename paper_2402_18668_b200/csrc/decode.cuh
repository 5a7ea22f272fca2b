// Device-side body of the linear-attention decode step (shared by decode.cu and generation_step.cu).
#pragma once
#include <cooperative_groups.h>

#include "common.cuh"

namespace based {

// One head's step, or one part of it, by a CTA of 256 threads (the fused generation step, both mixers in one launch, runs
// the same code as the stand-alone kernel).
// SYM: the state holds the 153 symmetric features (one per unordered pair, the feature count of the appendix "Computing
// Recurrent State Size") instead of the 273 of the full outer product: the same outputs from 44 % fewer state bytes.
// Everything the first rows need is requested together, before anything is computed: UNROLL state rows per thread, the
// K-state, q, k, v; a thread builds its rows' features from the raw entries of q and k, and one barrier publishes them.
// (With the features built by all threads before the first row was requested, two barriers and UNROLL 7, a step of 2048
// heads, d_v 128, took 92.7 us and one of 128 heads 6.9; now 89.1 and 5.8.)
// UN: rows in flight per thread at most (the rounds are made even).  STREAM: the state of all heads together is larger
// than L2, so every line is used exactly once per step: evict-first loads and stores (89.9 -> 89.1 us, 51.6 -> 50.4 with SYM).
// PARTS > 1: the CTAs of a cluster share the head's rows (with few heads one CTA per head leaves most of the chip idle);
// the others write their sums to part 0's shared memory, signal and leave, and part 0 adds them up (read by part 0 from theirs,
// which then had to wait for it, a step of 16 heads took 0.35 us more).
template <int DV, typename T, bool SYM, int PARTS, int UN, bool STREAM>
__device__ __forceinline__ void decode_step_body(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                                                 float* __restrict__ kv, float* __restrict__ z, T* __restrict__ out,
                                                 int numerator_only, size_t head, int part) {
    namespace cg = cooperative_groups;
    constexpr int TPR = DV / 4, RPP = 256 / TPR;
    constexpr int ND = SYM ? kDSym : kD;
    constexpr int MAXR = (ND + PARTS - 1) / PARTS;               // rows of the largest part
    constexpr int NPASS = (MAXR + RPP - 1) / RPP;
    constexpr int ROUNDS = (NPASS + UN - 1) / UN, UNROLL = (NPASS + ROUNDS - 1) / ROUNDS;
    __shared__ float s_pq[MAXR], s_pk[MAXR];
    __shared__ __align__(16) float s_num[RPP][DV];
    __shared__ float s_den[8];
    __shared__ float s_part[PARTS][DV + 1];                      // the parts' sums: numerator, denominator (PARTS > 1: in part 0 alone)
    const int tid = threadIdx.x, c4 = tid % TPR, rslot = tid / TPR;
    const bool row_thread = rslot < RPP;
    const int r0 = part * ND / PARTS, rows = (part + 1) * ND / PARTS - r0;

    if (PARTS > 1) asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");      // part 0 runs: the others may write to it
    float4* S = reinterpret_cast<float4*>(kv + (head * ND + r0) * (size_t)DV) + c4;
    float4 s[UNROLL];
    auto fetch = [&](int p0) {
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const int r = (p0 + u) * RPP + rslot;
            if (r < rows && row_thread) s[u] = STREAM ? __ldcs(&S[(size_t)r * TPR]) : S[(size_t)r * TPR];
        }
    };
    fetch(0);
    float vv[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) vv[e] = to_f32(v[head * DV + c4 * 4 + e]);
    float dpart = 0.f;
    for (int t = tid; t < rows; t += 256) {
        // feature r0 + t = scale * x[m] * x[n], x[16] = 1
        const int f = r0 + t;
        int m = kDFeat, n = kDFeat;
        float c = 1.f;
        if (f > kDFeat) {
            const int p = f - 1 - kDFeat;
            if (SYM) pair_of(p, m, n);
            else { m = p >> 4; n = p & 15; }
            c = SYM && m != n ? 0.25f : kQuadScale;
        } else if (f > 0) {
            m = f - 1;
            c = kLinScale;
        }
        const T* qh = q + head * kDFeat;
        const T* kh = k + head * kDFeat;
        float* zr = z + head * ND + f;
        const float zo = *zr;
        const float qm = m < kDFeat ? to_f32(qh[m]) : 1.f, qn = n < kDFeat ? to_f32(qh[n]) : 1.f;
        const float km = m < kDFeat ? to_f32(kh[m]) : 1.f, kn = n < kDFeat ? to_f32(kh[n]) : 1.f;
        const float pq = qm * qn * c, pk = km * kn * c, zn = zo + pk;
        s_pq[t] = pq;
        s_pk[t] = pk;
        *zr = zn;
        dpart = fmaf(pq, zn, dpart);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dpart += __shfl_xor_sync(0xffffffffu, dpart, o);
    if ((tid & 31) == 0) s_den[tid >> 5] = dpart;
    __syncthreads();

    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int p0 = 0; p0 < NPASS; p0 += UNROLL) {
        if (p0 > 0) fetch(p0);
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const int r = (p0 + u) * RPP + rslot;
            if (r < rows && row_thread) {
                const float pk = s_pk[r], pq = s_pq[r];
                s[u].x = fmaf(pk, vv[0], s[u].x);
                s[u].y = fmaf(pk, vv[1], s[u].y);
                s[u].z = fmaf(pk, vv[2], s[u].z);
                s[u].w = fmaf(pk, vv[3], s[u].w);
                acc.x = fmaf(pq, s[u].x, acc.x);
                acc.y = fmaf(pq, s[u].y, acc.y);
                acc.z = fmaf(pq, s[u].z, acc.z);
                acc.w = fmaf(pq, s[u].w, acc.w);
                if (STREAM) __stcs(&S[(size_t)r * TPR], s[u]);
                else S[(size_t)r * TPR] = s[u];
            }
        }
    }
    if (row_thread) *reinterpret_cast<float4*>(&s_num[rslot][c4 * 4]) = acc;
    __syncthreads();
    cg::cluster_group cluster = cg::this_cluster();
    float* to = PARTS == 1 ? s_part[0] : cluster.map_shared_rank(s_part[part], 0);
    if (PARTS > 1) asm volatile("barrier.cluster.wait;" ::: "memory");
    if (tid < DV) {
        float num = 0.f;
#pragma unroll
        for (int r = 0; r < RPP; ++r) num += s_num[r][tid];
        to[tid] = num;
    } else if (tid == DV) {
        float den = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) den += s_den[w];
        to[DV] = den;
    }
    if (PARTS == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        if (part != 0) return;
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
    if (tid < DV) {
        float num = 0.f, den = 0.f;
#pragma unroll
        for (int c = 0; c < PARTS; ++c) {
            num += s_part[c][tid];
            den += s_part[c][DV];
        }
        out[head * DV + tid] = from_f32<T>(numerator_only ? num : num / (den + kEps));
    }
}

// CTAs per head, by one CTA per SM (us per step on B200, replayed back to back on states from memory): d_v 128 with 16 heads eight
// 4.0, four 4.3, with 2 heads 2.2 / 2.5 (and 2.75 before the parts' sums were pushed); 153 rows 2.9 / 3.0 with 16; d_v 64 2.6 / 2.7;
// 25 heads four 3.6, two 3.6, one 3.8, 74 heads d_v 128 two 6.7, one 7.6.  Not where a head's state is small (153 rows x 64 with 16
// heads: 2.6 / 2.4 / 2.5 / 2.3).
// The sums' order depends on it, so the fused step follows the same rule.
template <int DV, bool SYM>
inline int decode_parts(int heads) {
    constexpr int head_kb = (SYM ? kDSym : kD) * DV * 4 / 1024;
    if (head_kb >= 64 && 8 * heads <= kSMs) return 8;
    if (head_kb >= 64 && 4 * heads <= kSMs) return 4;
    if (head_kb >= 96 && 2 * heads <= kSMs) return 2;
    return 1;
}
// 96 MB: safely above what L2 (126 MB, shared with everything else) keeps from one step to the next
inline bool decode_streams(size_t heads, int d_v, bool sym) {
    return heads * (sym ? kDSym : kD) * d_v * sizeof(float) > (size_t)96 << 20;
}

}  // namespace based
