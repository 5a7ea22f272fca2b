// Forward of the definition form (left-hand side of Eq. (2) of Sec. 4.1) on the tensor cores, bf16 io, empty initial state, for the
// feature dimensions 8, 24 and 32, which the chunked d' = 16 kernel does not cover, and for one chunk of d' = 16 without a state:
//   out = (sum_j w_ij v_j) / (sum_j w_ij + eps),  w = 1 + s/sqrt(d') + s^2/(2 d'),  s = q_i . k_j.
//
// One CTA per (head, 128 queries), looping over tiles of 64 keys: S = Q K^T to tensor memory, the rows' threads turn it into weights
// (bf16, over the scores; row sums of the unrounded ones in registers), Y += W V with the weights as they lie.  Eleven warps, two
// CTAs per SM: two groups of four row warps that take the key tiles in turn, one warp each for the scores' MMAs, the products'
// MMAs and the loads.  Three sets of score columns (two at d_v 128): the scores of the next tiles are there when a group comes
// for them, so that what a row warp waits for is its own arithmetic.  Against one group and one set of scores per CTA and four (d_v
// 128, then: two) CTAs per SM (backward_tc.cu, kModeFwd): at d_v 128, where a second set was missing most, 59 -> 49 us at d' 32 B4 H16
// L2048 and 216 -> 164 at d' 24 L4096; with a head alone 20 -> 12 (L2048 d_v 64).  At d_v 64 with every SM busy the two are the same:
// half of the issue slots are used, 1075 warp instructions per tile of 128 x 64 pairs.  A row warp loads sixteen score columns ahead
// of the ones it works on: d_v 128 d' 24 47.8 -> 46.9, 64 heads L777 16.7 -> 16.2.  What bounds it is no single part (64 heads L8192 d_v
// 64, 431 us, parts left out: the rows' work 327, the scores 398, the products 348, both 326, all three 281, the loads too 182): the
// hand-overs of a tile, and 11 KB of loads for it.  A third row group changes nothing, nor do eight stages for six; 256 queries a CTA,
// each key tile loaded for two halves, gains 8 % there and loses 5 at L2048 (38 us) and half at few heads.
#include <math.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "sm100.cuh"

namespace based {
using namespace sm100;

namespace {
constexpr int kOwnQ = 128, kLTQ = 64, kThreadsQ = 352;

template <int DV> struct FCfg {
    static constexpr int kVB = (DV + 63) / 64;                         // 64-column blocks of a v tile
    static constexpr int kNSet = DV == 64 ? 3 : 2, kNS = DV == 64 ? 6 : 4;
    // shared memory: q [128][32] and k [64][32] (columns past d' are zero), 64-byte rows, SWIZZLE_64B; v [kVB][64][64], SWIZZLE_128B
    static constexpr uint32_t kNarrow = kLTQ * 64, kStage = kNarrow + kVB * kLTQ * 128;
    static constexpr uint32_t offStage = kOwnQ * 64, offDen = offStage + kNS * kStage, offBars = offDen + 2 * kOwnQ * 4;
    static constexpr uint32_t kSmem = offBars + 512 + 1024;
    static constexpr uint32_t colY = kNSet * kLTQ;
    static_assert(colY + 64 * kVB <= 256 && 2 * (kSmem + 1024) <= 228 * 1024, "two CTAs per SM");
    static_assert(kNS * kStage >= (uint32_t)kVB * kOwnQ * 128, "the output tile fits the stages");
};
enum { qOwn = 0, qFull = 1, qEmpty = 7, qScore = 13, qWeight = 16, qFree = 19, qFinal = 22, qCount = 23 };

struct FParams {
    unsigned int* err;
    int heads, L, dvw, numerator_only, kdim, by_length, overlapped;
    float s1, s2;                                                      // w = 1 + s s1 + s^2 s2
};

__device__ __forceinline__ uint64_t pair_of_f(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void halves_of(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma_pairs(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add_pairs(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}
// AND over the row threads; orders their shared-memory accesses
__device__ __forceinline__ bool all_rows(bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, 256, p;\n\t"
        "selp.b32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)pred)
        : "memory");
    return r != 0;
}
}  // namespace

// IN_ORDER: one chunk of d' 16.  The first group takes both key tiles, and a row's weights are summed as the chunked kernel sums them
// (the even columns, the odd ones, then both; so does kModeFwd), so that the outputs are the bits that the chunked kernel gives beside a
// state (us, both groups / this: L128, 16 heads d_v 64 3.24 / 3.36, d_v 128 3.72 / 3.82, 200 heads d_v 128 5.18 / 5.01, 400 8.34 / 8.43).
// At d_v 64 the rounded weights, as there (prefill_tc_kernel's ROUNDED): 16 heads L128 3.66 -> 3.81, 600 8.6 -> 9.0.
template <int DV, bool IN_ORDER>
__global__ void __launch_bounds__(kThreadsQ, 2)
    quadratic_fwd_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                            const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_out, const FParams p) {
    using C = FCfg<DV>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::offBars);
    uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(bars + qCount);
    volatile uint32_t* abort_flag = tmem_base_s + 1;
    float* s_den = reinterpret_cast<float*>(smem + C::offDen);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ntiles = (p.L + kOwnQ - 1) / kOwnQ;
    const int turn = p.by_length ? blockIdx.x / p.heads : blockIdx.x % ntiles;
    const int head = p.by_length ? blockIdx.x - turn * p.heads : blockIdx.x / ntiles;
    const int r0 = (ntiles - 1 - turn) * kOwnQ;                        // the longest loops first
    const int n = (min(p.L, r0 + kOwnQ) - 1) / kLTQ + 1;

    if (tid == 0) {
        mbar_init(&bars[qOwn], 1);
        mbar_init(&bars[qFinal], 1);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            mbar_init(&bars[qFull + i], 1);
            mbar_init(&bars[qEmpty + i], 1);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            mbar_init(&bars[qScore + i], 1);
            mbar_init(&bars[qWeight + i], 128);
            mbar_init(&bars[qFree + i], 1);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 8) {
        tmem_alloc(tmem_base_s, 256);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = *tmem_base_s;
    bool ok = true;
    // (a dependent launch: alone, or beside the state's kernel, which has waited for what is ahead of both)
    if (!p.overlapped) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 8 || warp == 9) {
        // ============================================================================ MMA warps: scores, products
        constexpr uint64_t dN = make_smem_desc_base(16, 512, kSwizzle64B);
        constexpr uint64_t dV = make_smem_desc_base(kLTQ * 128, 1024, kSwizzle128B);
        constexpr uint32_t iS = make_idesc_bf16(128, kLTQ, 0, 0), iY = make_idesc_bf16(128, 64 * C::kVB, 0, 1);
        const uint32_t lead = elect_one();
        const uint32_t aQ = smem_u32(smem) >> 4;
        auto stage_at = [&](int t) { return smem_u32(smem + C::offStage + (t % C::kNS) * C::kStage) >> 4; };
        if (warp == 8) {
            ok = mbar_wait(&bars[qOwn], 0, abort_flag);
            for (int t = 0; t < n && ok; ++t) {
                const int set = t % C::kNSet;
                ok = mbar_wait(&bars[qFull + t % C::kNS], (t / C::kNS) & 1, abort_flag) &&
                     (t < C::kNSet || mbar_wait(&bars[qFree + set], (t / C::kNSet - 1) & 1, abort_flag));
                if (!ok) break;
                tc_fence_after();
                const uint32_t d = tb + set * kLTQ, aK = stage_at(t);
                mma_ss_w<false>(lead, d, desc_lo(dN) + aQ, desc_hi(dN), desc_lo(dN) + aK, desc_hi(dN), iS);
                if (p.kdim > 16) mma_ss_w<true>(lead, d, desc_lo(dN) + aQ + 2, desc_hi(dN), desc_lo(dN) + aK + 2, desc_hi(dN), iS);
                mma_commit_w(lead, &bars[qScore + set]);
            }
        } else {
            for (int t = 0; t < n && ok; ++t) {
                const int set = t % C::kNSet;
                ok = mbar_wait(&bars[qWeight + set], (t / C::kNSet) & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                const uint32_t aV = stage_at(t) + (C::kNarrow >> 4);
#pragma unroll
                for (int k = 0; k < kLTQ / 16; ++k) {
                    const uint32_t a = tb + set * kLTQ + 8 * k, b = desc_lo(dV) + aV + 128 * k;
                    if (k == 0 && t == 0) mma_ts_w<false>(lead, tb + C::colY, a, b, desc_hi(dV), iY);
                    else mma_ts_w<true>(lead, tb + C::colY, a, b, desc_hi(dV), iY);
                }
                mma_commit_w(lead, &bars[qFree + set]);
                mma_commit_w(lead, &bars[qEmpty + t % C::kNS]);
            }
            if (ok) mma_commit_w(lead, &bars[qFinal]);
        }
    } else if (warp == 10) {
        // ============================================================================ loads
        const uint32_t lead = elect_one();
        if (lead) {
            mbar_arrive_expect_tx(&bars[qOwn], kOwnQ * 64);
            tma_load_3d(smem, &tm_q, &bars[qOwn], 0, r0, head);
        }
        for (int t = 0; t < n && ok; ++t) {
            const int s = t % C::kNS;
            if (t >= C::kNS) ok = mbar_wait(&bars[qEmpty + s], (t / C::kNS - 1) & 1, abort_flag);
            if (!ok || !lead) continue;
            uint8_t* st = smem + C::offStage + s * C::kStage;
            mbar_arrive_expect_tx(&bars[qFull + s], C::kStage);
            tma_load_3d(st, &tm_k, &bars[qFull + s], 0, t * kLTQ, head);
#pragma unroll
            for (int b = 0; b < C::kVB; ++b)
                tma_load_3d(st + C::kNarrow + b * (kLTQ * 128), &tm_v, &bars[qFull + s], b * 64, t * kLTQ, head);
        }
    } else {
        // ============================================================================ rows
        const int wg = warp >> 2, row_l = tid & 127, row = r0 + row_l;
        const uint32_t lane_base = (uint32_t)(warp & 3) * 32u;
        const int rw = r0 + (int)lane_base;
        const uint64_t k1 = pair_of_f(p.s1, p.s1), k2 = pair_of_f(p.s2, p.s2), one = pair_of_f(1.f, 1.f);
        uint64_t den2[2] = {0, 0};
        // 16 scores to weights, packed in pairs from w[w0] on; first: the masked form's first column
        auto weights = [&](auto masked_tag, const uint32_t (&sr)[16], uint32_t (&w)[16], int w0, int first) {
            constexpr bool MASKED = decltype(masked_tag)::value;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint64_t s = pair_of_f(__uint_as_float(sr[2 * i]), __uint_as_float(sr[2 * i + 1]));
                uint64_t x = fma_pairs(s, fma_pairs(s, k2, k1), one);
                float lo, hi;
                if (MASKED) {
                    const int col = first + 2 * i;
                    halves_of(x, lo, hi);
                    x = pair_of_f(col <= row ? lo : 0.f, col + 1 <= row ? hi : 0.f);
                }
                halves_of(x, lo, hi);
                const uint32_t packed = pack2(lo, hi);
                w[w0 + i] = packed;
                uint64_t& den = den2[IN_ORDER ? 0 : i & 1];
                den = add_pairs(den, IN_ORDER && DV == 64 ? pair_of_f(__uint_as_float(packed << 16), __uint_as_float(packed & 0xffff0000u)) : x);
            }
        };
        // (what was loaded is used behind its wait and not before it)
        auto landed = [&](uint32_t (&r)[16]) {
            tmem_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) asm volatile("" : "+r"(r[i]));
        };
        uint32_t s0[16], s1[16], w[16];
        for (int t = !IN_ORDER ? wg : wg == 0 ? 0 : n; t < n; t += IN_ORDER ? 1 : 2) {
            const int si = t % C::kNSet;
            const uint32_t set = tmem_addr(tb, lane_base, si * kLTQ);
            ok = __all_sync(~0u, mbar_wait(&bars[qScore + si], (t / C::kNSet) & 1, abort_flag));
            if (!ok) break;
            tc_fence_after();
            if (t * kLTQ + kLTQ <= rw) {
                // sixteen columns at a time, the next ones' load under way; the weights go over columns read before
                tmem_ld16(set, s0);
                landed(s0);
                tmem_ld16(set + 16, s1);
                weights(std::false_type{}, s0, w, 0, 0);
                landed(s1);
                tmem_ld16(set + 32, s0);
                weights(std::false_type{}, s1, w, 8, 0);
                tmem_st16(set, w);
                landed(s0);
                tmem_ld16(set + 48, s1);
                weights(std::false_type{}, s0, w, 0, 0);
                landed(s1);
                weights(std::false_type{}, s1, w, 8, 0);
                tmem_st16(set + 16, w);
            } else {
#pragma unroll 1
                for (int h = 0; h < 2; ++h) {
                    const int cb = t * kLTQ + 32 * h;
                    if (cb > rw) {                                     // no live pair
#pragma unroll
                        for (int e = 0; e < 16; ++e) w[e] = 0u;
                    } else {
                        tmem_ld16(set + 32 * h, s0);
                        tmem_ld16(set + 32 * h + 16, s1);
                        landed(s0);
                        landed(s1);
                        weights(std::true_type{}, s0, w, 0, cb);
                        weights(std::true_type{}, s1, w, 8, cb + 16);
                    }
                    tmem_st16(set + 16 * h, w);
                }
            }
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(&bars[qWeight + si]);
        }
        float a, b;
        halves_of(add_pairs(den2[0], den2[1]), a, b);
        s_den[wg * kOwnQ + row_l] = a + b;
        ok = all_rows(ok && mbar_wait(&bars[qFinal], 0, abort_flag));
        tc_fence_after();
        if (ok) {
            // half of the columns each, scaled, in the layout of a TMA box (128-byte rows, SWIZZLE_128B) over the stages, and out by TMA
            const float sc = p.numerator_only ? 1.0f : 1.0f / (s_den[row_l] + s_den[kOwnQ + row_l] + kEps);
            uint8_t* out_s = smem + C::offStage;
            for (int c = wg * (DV / 32); c < (wg + 1) * (DV / 32); ++c) {
                uint32_t r[16];
                tmem_ld16(tmem_addr(tb, lane_base, C::colY + 16 * c), r);
                tmem_wait_ld();
                uint32_t o[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) o[e] = pack2(__uint_as_float(r[2 * e]) * sc, __uint_as_float(r[2 * e + 1]) * sc);
                uint8_t* rowp = out_s + (c >> 2) * (kOwnQ * 128) + row_l * 128;
                *reinterpret_cast<uint4*>(rowp + ((((2 * c) & 7) ^ (row_l & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
                *reinterpret_cast<uint4*>(rowp + ((((2 * c + 1) & 7) ^ (row_l & 7)) << 4)) = make_uint4(o[4], o[5], o[6], o[7]);
            }
            fence_proxy_async_smem();
            all_rows(true);
            if (tid == 0) {
#pragma unroll
                for (int bb = 0; bb < C::kVB; ++bb) tma_store_3d(&tm_out, out_s + bb * (kOwnQ * 128), bb * 64, r0, head);
                tma_store_commit();
                tma_store_wait_read<0>();
            }
        }
    }
    if (!ok && lane == 0) atomicOr(p.err, 1u);
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);     // loads still in flight get time to land
    }
    __syncthreads();
    if (warp == 8) tmem_dealloc(tb, 256);
    // one CTA holds the grid's end back until the grid before it is complete: what follows in the stream sees both
    if (p.overlapped && blockIdx.x == gridDim.x - 1 && tid == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
}

namespace {
template <int DV, bool IN_ORDER>
based_status launch_forward(const CUtensorMap& q, const CUtensorMap& k, const CUtensorMap& v, const CUtensorMap& out, const FParams& p,
                            unsigned grid, cudaStream_t stream) {
    using C = FCfg<DV>;
    {
        static bool configured[64] = {};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BASED_ERR_CUDA;
        std::lock_guard<std::mutex> lock(setup_mutex());
        if (!configured[dev]) {
            if (cudaFuncSetAttribute(quadratic_fwd_tc_kernel<DV, IN_ORDER>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::kSmem) != cudaSuccess)
                return BASED_ERR_CUDA;
            configured[dev] = true;
        }
    }
    const cudaError_t e = launch_ex(quadratic_fwd_tc_kernel<DV, IN_ORDER>, dim3(grid), dim3(kThreadsQ), C::kSmem, 1,
                                    p.overlapped || dependent_forward(grid, grid / p.heads, 2 * kSMs), stream, q, k, v, out, p);
    note_launch();
    const based_status st = check_launch("quadratic_fwd_tc_kernel");
    return e == cudaSuccess ? st : BASED_ERR_CUDA;
}
}  // namespace

based_status launch_quadratic_groups_tc(const void* q, const void* k, const void* v, void* out, int BH, int L,
                                        int d_feat, int d_v, int numerator_only, bool overlapped, cudaStream_t stream) {
    CUtensorMap tq, tk, tv, to;
    const CUtensorMapSwizzle s64 = CU_TENSOR_MAP_SWIZZLE_64B, s128 = CU_TENSOR_MAP_SWIZZLE_128B;
    if (!make_rows_map_bf16(&tq, q, BH, L, d_feat, 32, kOwnQ, s64) || !make_rows_map_bf16(&tk, k, BH, L, d_feat, 32, kLTQ, s64) ||
        !make_rows_map_bf16(&tv, v, BH, L, d_v, 64, kLTQ, s128) || !make_rows_map_bf16(&to, out, BH, L, d_v, 64, kOwnQ, s128))
        return BASED_ERR_CUDA;
    FParams p{};
    if (error_word_ptr(&p.err) != BASED_OK) return BASED_ERR_CUDA;
    p.heads = BH;
    p.L = L;
    p.dvw = d_v;
    p.numerator_only = numerator_only;
    p.kdim = d_feat <= 16 ? 16 : 32;
    p.s1 = 1.0f / sqrtf((float)d_feat);
    p.s2 = 0.5f / (float)d_feat;
    p.overlapped = overlapped;
    const long long ctas = (long long)((L + kOwnQ - 1) / kOwnQ) * BH;
    p.by_length = ctas > kSMs;
    const bool in_order = d_feat == kDFeat;
    if (d_v == 64) return in_order ? launch_forward<64, true>(tq, tk, tv, to, p, (unsigned)ctas, stream) : launch_forward<64, false>(tq, tk, tv, to, p, (unsigned)ctas, stream);
    return in_order ? launch_forward<128, true>(tq, tk, tv, to, p, (unsigned)ctas, stream) : launch_forward<128, false>(tq, tk, tv, to, p, (unsigned)ctas, stream);
}

}  // namespace based
