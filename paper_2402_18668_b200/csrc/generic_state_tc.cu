// based_prefill for the feature dimensions 8, 24 and 32 (bf16 io): the final recurrent state
// (Sec. 4.1, Eq. (3): S = sum_j phi(k_j) v_j^T, z = sum_j phi(k_j)) on the tensor cores.
//
//   S[f, :] (+)= sum_j phi_f(k_j) v_j        z[f] (+)= sum_j phi_f(k_j)
//
// Rows of the state: row 0 constant, rows 1..d' linear, row 1 + d' + m d' + n the product k_m k_n.  Rows (m, n) and (n, m)
// are equal, so one feature per unordered pair is summed and stored twice.  The features, in the operand's order:
// f < d': k_f | d' + d' o + m, o < d' / 2: k_m k_(m + o mod d') | then k_m k_(m + d' / 2), m < d' / 2 | then 1.
//
// One CTA per (head, part of FN features), 288 threads: two groups of four row warps take every second step of 64 tokens,
// warp 8 (converged, one elected lane) issues TMA loads and MMAs.  Two row threads per token hold its k row in registers,
// two values a word, form half of the part's features each as packed bf16 products (a pair of features per instruction: with
// the order above their factors are neighbours) and write them as the token's row of the B operand, [64 tokens][FN],
// MN-major, SWIZZLE_32B blocks of 16 features.  The value tile comes by TMA and is the A operand as it lies ([64 tokens]
// [d_v], MN-major), so the accumulator in tensor memory is the transposed state, [d_v lanes][FN columns] fp32: at the end a
// warp stores 128 consecutive bytes of a state row per feature.  z: rows of ones below the values, lanes 64 on of the same
// accumulator at d_v 64, an accumulator of its own (M = 64) at d_v 112 / 128.  The feature scales 1 / d'^(1/4) and
// 1 / (sqrt 2 sqrt d') multiply the fp32 sums at the end, so the operand carries one rounding (of the product) only.
// Bound: the MMAs' operand reads (a burst of four takes 480 cycles at d' 24 d_v 64, 176 of them arithmetic) and the chain of
// a group's wait, write and hand-over beside them; the rows two steps ahead instead of one change nothing.  An accumulator
// lane per feature instead, whose thread read both factors of 64 tokens from a transposed k tile, took three times the
// shared-memory traffic and loaded the value tile once per 128 features: B4 H16 L2048 d_v 64 at d' 8 / 24 / 32 22.7 / 40.5 /
// 56.1 us, here 12.6 / 16.1 / 25.6; d_v 128 d' 24 50 -> 27; B1 H8 L300 d' 24 8.9 -> 6.9 (with the sums stored straight from
// tensor memory, a state row's number per element, 24.5 and 15.1).  d' 32 in three parts of 192, two waves: 30.4.
#include <cuda_bf16.h>
#include <math.h>

#include <mutex>
#include <type_traits>
#include <utility>

#include "common.cuh"
#include "sm100.cuh"

namespace based {
using namespace sm100;

namespace {
constexpr int kTB = 64;            // tokens per step (K extent of one MMA burst)
constexpr int kRowThreads = 256;   // two groups of four row warps
constexpr int kThreadsS = kRowThreads + 32;    // and the issuer warp

template <int DF, int DV> struct SCfg {
    static constexpr int kNF = 1 + DF + DF * (DF + 1) / 2;     // features: one per unordered pair
    // features per CTA: as few parts as the accumulators fit 256 tensor-memory columns in (d_v 128: two of them)
    static constexpr int kFN = DF == 8 ? 48 : DF == 24 ? (DV == 64 ? 176 : 112) : (DV == 64 ? 144 : 128);
    static constexpr int kParts = (kNF + kFN - 1) / kFN;
    static constexpr int kVB = (DV + 63) / 64;                 // 64-column blocks of the v tile (112 -> 2)
    static constexpr int kNS = DV == 64 ? 4 : 3;               // load stages
    static constexpr uint32_t kVBytes = kVB * kTB * 128;       // [64 tokens][64 * kVB] bf16, SWIZZLE_128B blocks
    static constexpr uint32_t kPhiBlk = kTB * 32;              // [64 tokens][16 features]
    static constexpr uint32_t kPhiBytes = (kFN / 16) * kPhiBlk;
    static constexpr uint32_t offPhi = kNS * kVBytes;          // two buffers, one per row group
    static constexpr uint32_t offOnes = (offPhi + 2 * kPhiBytes + 1023) / 1024 * 1024;   // 16 tokens x 64 columns of ones (A operand of z)
    static constexpr uint32_t offMisc = offOnes + 2048;
    static constexpr uint32_t kSmem = offMisc + 256 + 1024;
    static constexpr uint32_t colZ = DV == 64 ? 0 : kFN;       // d_v 64: lanes 64 on of the state's columns
    static constexpr uint32_t kColsUsed = DV == 64 ? kFN : 2 * kFN;
    static constexpr uint32_t kCols = kColsUsed <= 64 ? 64 : kColsUsed <= 128 ? 128 : 256;
    static_assert(kColsUsed <= 256 && kFN % 16 == 0 && kFN <= kRowThreads, "tensor memory budget");
    static_assert(kFN * (DV + 1) * 4 <= (int)offOnes, "the sums' way out");
};
enum { sFull0 = 0, sAlu0 = 4, sMma0 = 6, sFinal = 8, sNum = 9 };

struct SParams {
    const __nv_bfloat16* k;        // [BH, L, d']
    float* kv;                     // [BH, D, dvw]
    float* z;                      // [BH, D]
    unsigned int* err;
    int L, dvw, cont;
    float lin, quad;
};
// AND of a predicate over the row threads (named barrier 2); also a barrier for their shared-memory traffic
__device__ __forceinline__ bool rows_and(bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 2, %2, p;\n\t"
        "selp.b32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)pred), "n"(kRowThreads)
        : "memory");
    return r != 0;
}
// f(i) with i as a constant, i one of I...
template <class F, int... I> __device__ __forceinline__ void pick(int i, F& f, std::integer_sequence<int, I...>) {
    ((i == I ? f(std::integral_constant<int, I>{}) : (void)0), ...);
}
}  // namespace

template <int DF, int DV>
__global__ void __launch_bounds__(kThreadsS, 2)
    generic_state_tc_kernel(const __grid_constant__ CUtensorMap tm_v, const SParams p) {
    using C = SCfg<DF, DV>;
    constexpr int FN = C::kFN, kD = 1 + DF + DF * DF;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::offMisc);
    uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(bars + sNum);
    volatile uint32_t* abort_flag = tmem_base_s + 1;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int head = blockIdx.y, part = blockIdx.x;
    const int nit = (p.L + kTB - 1) / kTB;

    if (tid == 0) {
        for (int s = 0; s < C::kNS; ++s) mbar_init(&bars[sFull0 + s], 1);
        for (int b = 0; b < 2; ++b) { mbar_init(&bars[sAlu0 + b], kRowThreads / 2); mbar_init(&bars[sMma0 + b], 1); }
        mbar_init(&bars[sFinal], 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    for (int i = tid; i < 512; i += kThreadsS) reinterpret_cast<uint32_t*>(smem + C::offOnes)[i] = 0x3f803f80u;
    fence_proxy_async_smem();
    if (warp == 8) { tmem_alloc(tmem_base_s, C::kCols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = *tmem_base_s;
    bool ok = true;
    // A dependent launch: set up while the grid ahead drains.  The outputs' kernel, if one follows, needs nothing of this one: it may
    // take what SMs have left once that grid is complete.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 8) {
        // the whole warp runs this block; one elected lane issues the MMAs, commits and loads (see mma_ss_w)
        const uint32_t lead = elect_one();
        constexpr uint64_t dPhi = make_smem_desc_base(C::kPhiBlk, 256, kSwizzle32B);      // B, MN-major: 16-feature blocks
        constexpr uint64_t dV = make_smem_desc_base(kTB * 128, 1024, kSwizzle128B);       // A, MN-major: 64-column blocks
        constexpr uint32_t iS = make_idesc_bf16(128, FN, 1, 1);
        constexpr uint32_t iZ = make_idesc_bf16(64, FN, 1, 1);
        const uint32_t aOnes = smem_u32(smem + C::offOnes);
        auto load = [&](int it) {
            if (!lead) return;
            const int s = it % C::kNS;
            uint8_t* st = smem + s * C::kVBytes;
            mbar_arrive_expect_tx(&bars[sFull0 + s], C::kVBytes);
#pragma unroll
            for (int b = 0; b < C::kVB; ++b)
                tma_load_3d(st + b * (kTB * 128), &tm_v, &bars[sFull0 + s], b * 64, it * kTB, head);
        };
        for (int it = 0; it < C::kNS && it < nit; ++it) load(it);
        for (int it = 0; it < nit && ok; ++it) {
            const int b = it & 1, s = it % C::kNS;
            ok = mbar_wait(&bars[sFull0 + s], (it / C::kNS) & 1, abort_flag);
            if (!ok) break;
            ok = mbar_wait(&bars[sAlu0 + b], (it >> 1) & 1, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const uint32_t aV = smem_u32(smem + s * C::kVBytes);
            const uint32_t lPhi = desc_lo(dPhi) + (smem_u32(smem + C::offPhi + b * C::kPhiBytes) >> 4);
#pragma unroll
            for (int kk = 0; kk < kTB / 16; ++kk) {
                const uint32_t aK = aV + kk * 2048;          // sixteen tokens on
                // d_v 64: rows 0..63 of A from the value tile, rows 64..127 from the ones
                const uint64_t dA = DV == 64 ? make_smem_desc_base(aOnes - aK, 1024, kSwizzle128B) : dV;
                const uint32_t a_lo = desc_lo(dA) + (aK >> 4), a_hi = desc_hi(dA);
                if (it == 0 && kk == 0) mma_ss_w<false>(lead, tb, a_lo, a_hi, lPhi + kk * 32, desc_hi(dPhi), iS);
                else mma_ss_w<true>(lead, tb, a_lo, a_hi, lPhi + kk * 32, desc_hi(dPhi), iS);
                if (DV != 64) {
                    const uint32_t o_lo = desc_lo(dV) + (aOnes >> 4);
                    if (it == 0 && kk == 0) mma_ss_w<false>(lead, tb + C::colZ, o_lo, desc_hi(dV), lPhi + kk * 32, desc_hi(dPhi), iZ);
                    else mma_ss_w<true>(lead, tb + C::colZ, o_lo, desc_hi(dV), lPhi + kk * 32, desc_hi(dPhi), iZ);
                }
            }
            mma_commit_w(lead, &bars[sMma0 + b]);
            // the previous step's products are done long since: its stage takes the load kNS steps ahead
            if (it >= 1 && it - 1 + C::kNS < nit) {
                ok = mbar_wait(&bars[sMma0 + ((it - 1) & 1)], ((it - 1) >> 1) & 1, abort_flag);
                if (!ok) break;
                load(it - 1 + C::kNS);
            }
        }
        if (ok) mma_commit_w(lead, &bars[sFinal]);
    } else {
        // ===================================================================== row threads
        constexpr int NW = DF / 2, kPc = FN / 8;             // words of a k row; 16-byte pieces of an operand row
        const int grp = tid >> 7, half = (tid >> 6) & 1;     // row group: every second step; half of the pieces
        const int t = tid & 63;                              // token of the step
        const uint32_t swz = (uint32_t)((t >> 2) & 1);
        uint8_t* prow = smem + C::offPhi + grp * C::kPhiBytes + t * 32;
        uint4 nx[NW / 4];                                    // the row of the group's next step
        auto fetch = [&](int it) {
            const int tok = it * kTB + t;
#pragma unroll
            for (int i = 0; i < NW / 4; ++i)
                nx[i] = it < nit && tok < p.L ? reinterpret_cast<const uint4*>(p.k + ((size_t)head * p.L + tok) * DF)[i]
                                              : make_uint4(0u, 0u, 0u, 0u);
        };
        fetch(grp);
        for (int it = grp; it < nit && ok; it += 2) {
            uint32_t xe[NW], xo[NW];                         // k_m, k_(m+1) with m even and odd
#pragma unroll
            for (int i = 0; i < NW / 4; ++i) {
                xe[4 * i] = nx[i].x; xe[4 * i + 1] = nx[i].y; xe[4 * i + 2] = nx[i].z; xe[4 * i + 3] = nx[i].w;
            }
#pragma unroll
            for (int i = 0; i < NW; ++i) xo[i] = __byte_perm(xe[i], xe[(i + 1) % NW], 0x5432);
            const uint32_t one = it * kTB + t < p.L ? 0x3f80u : 0u;      // past the end every feature vanishes
            fetch(it + 2);
            // the group's buffer is free once the products of two steps ago are done
            ok = __all_sync(~0u, it < 2 || mbar_wait(&bars[sMma0 + grp], ((it >> 1) - 1) & 1, abort_flag));
            if (!ok) break;
            auto pieces = [&](auto tag) {
                constexpr int H = decltype(tag)::value;      // 2 * part + half
                constexpr int l0 = (H & 1) ? (kPc + 1) / 2 : 0, l1 = (H & 1) ? kPc : (kPc + 1) / 2;
#pragma unroll
                for (int l = l0; l < l1; ++l) {
                    uint32_t pk[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int f = (H >> 1) * FN + l * 8 + 2 * i;
                        const int e = f - DF, m = f < DF ? f : e % DF;
                        const int n = (m + e / DF) % DF;     // the last group's offset is d' / 2
                        if (f >= C::kNF) pk[i] = 0u;
                        else if (f == C::kNF - 1) pk[i] = one;
                        else if (f < DF) pk[i] = xe[m / 2];
                        else asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(pk[i]) : "r"(xe[m / 2]), "r"(n & 1 ? xo[n / 2] : xe[n / 2]));
                    }
                    *reinterpret_cast<uint4*>(prow + (l >> 1) * C::kPhiBlk + (((l & 1) ^ swz) << 4)) =
                        make_uint4(pk[0], pk[1], pk[2], pk[3]);
                }
            };
            pick(2 * part + half, pieces, std::make_integer_sequence<int, 2 * C::kParts>{});         // warp-uniform
            fence_proxy_async_smem();
            mbar_arrive(&bars[sAlu0 + grp]);
        }
        ok = __all_sync(~0u, ok && mbar_wait(&bars[sFinal], 0, abort_flag));
        tc_fence_after();
        // Through shared memory, [FN features][d_v] fp32 in place of the stages and the operand (their products are done), so
        // that 16-byte words of a state row go out side by side and the rows' numbers are worked out once per word.
        float* sums = reinterpret_cast<float*>(smem);
        float* zsum = sums + FN * DV;
        if (ok) {                                            // warp-uniform: the loads are warp-collective
            const int quad = warp & 3, col = quad * 32 + lane;
            const uint32_t lane_base = (uint32_t)quad * 32u;
            for (int c = grp; c < FN / 16; c += 2) {
                uint32_t r[16];
                if (quad * 32 < DV) {
                    tmem_ld16(tmem_addr(tb, lane_base, c * 16), r);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i) sums[(c * 16 + i) * DV + col] = __uint_as_float(r[i]);
                }
                if (quad == (DV == 64 ? 2 : 0)) {            // every lane holds the same sums
                    tmem_ld16(tmem_addr(tb, lane_base, C::colZ + c * 16), r);
                    tmem_wait_ld();
                    if (lane == 0) {
#pragma unroll
                        for (int i = 0; i < 16; i += 4)
                            *reinterpret_cast<uint4*>(zsum + c * 16 + i) = make_uint4(r[i], r[i + 1], r[i + 2], r[i + 3]);
                    }
                }
            }
        }
        ok = rows_and(ok);
        if (ok) {
            // row of the state of a feature, and its twin: a pair's row (m, n) is the row (n, m) too
            auto rows = [&](int f, int& row, int& twin, float& scale) {
                const int e = f - DF, m = e % DF, n = (m + e / DF) % DF;
                const bool one = f == C::kNF - 1, lin = f < DF;
                row = one ? 0 : lin ? 1 + f : 1 + DF + m * DF + n;
                twin = one || lin ? row : 1 + DF + n * DF + m;
                scale = one ? 1.0f : lin ? p.lin : p.quad;
            };
            const size_t row0 = (size_t)head * kD;
            const int nf = min(FN, C::kNF - part * FN);
            constexpr int kQ = DV / 4;                       // 16-byte words of a row
            const int q4 = tid % kQ;
            for (int l = tid / kQ; l < nf && q4 * 4 < p.dvw; l += kRowThreads / kQ) {
                int row, twin;
                float scale;
                rows(part * FN + l, row, twin, scale);
                const float4 v = *reinterpret_cast<const float4*>(sums + l * DV + q4 * 4);
                float4* a = reinterpret_cast<float4*>(p.kv + (row0 + row) * p.dvw) + q4;
                float4* b = reinterpret_cast<float4*>(p.kv + (row0 + twin) * p.dvw) + q4;
                float4 oa = make_float4(v.x * scale, v.y * scale, v.z * scale, v.w * scale), ob = oa;
                if (p.cont) {
                    const float4 x = *a, y = *b;
                    oa.x += x.x; oa.y += x.y; oa.z += x.z; oa.w += x.w;
                    ob.x += y.x; ob.y += y.y; ob.z += y.z; ob.w += y.w;
                }
                *a = oa;
                if (twin != row) *b = ob;
            }
            if (tid < nf) {
                int row, twin;
                float scale;
                rows(part * FN + tid, row, twin, scale);
                const float o = zsum[tid] * scale;
                float* a = p.z + row0 + row;
                float* b = p.z + row0 + twin;
                const float x = p.cont ? *a : 0.f, y = p.cont ? *b : 0.f;
                *a = o + x;
                if (twin != row) *b = o + y;
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
    if (warp == 8) tmem_dealloc(tb, C::kCols);
}

namespace {
template <int DF, int DV>
based_status launch_state(const void* k, const void* v, float* kv, float* z, int BH, int L, int dvw, int cont,
                          cudaStream_t stream) {
    using C = SCfg<DF, DV>;
    CUtensorMap tv;
    if (!make_rows_map_bf16(&tv, v, BH, L, dvw, 64, kTB, CU_TENSOR_MAP_SWIZZLE_128B)) return BASED_ERR_CUDA;
    SParams p{};
    if (error_word_ptr(&p.err) != BASED_OK) return BASED_ERR_CUDA;
    p.k = static_cast<const __nv_bfloat16*>(k);
    p.kv = kv;
    p.z = z;
    p.L = L;
    p.dvw = dvw;
    p.cont = cont;
    const float rd = sqrtf((float)DF);
    p.lin = 1.0f / sqrtf(rd);
    p.quad = 1.0f / (1.41421356237309505f * rd);
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BASED_ERR_CUDA;
    {
        std::lock_guard<std::mutex> lock(setup_mutex());
        if (!configured[dev]) {
            if (cudaFuncSetAttribute(generic_state_tc_kernel<DF, DV>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)C::kSmem) != cudaSuccess)
                return BASED_ERR_CUDA;
            configured[dev] = true;
        }
    }
    // A dependent launch, but not at d' 32 with two tiles of values (five CTAs per head, the longest walks) where these CTAs would share the
    // SMs that the outputs' CTAs of a call before leave first, and each have one to itself behind the end of that call: too many of both for
    // the chip at once, but few outputs' tiles beyond (us repeated, dependent / plain, with the outputs, d_v 112: 16 heads L1409 24.5 /
    // 20.8, 24 L1024 19.6 / 17.4, 16 L2048 30.4 / 26.7, 10 L4096 52 / 45.6; d_v 128, dependent by plain: 20 L300 1.06, 18 L300 0.89, 32 L300
    // 0.95, 14 L1024 0.94, 20 L1024 1.11, 28 L1024 0.99, 13 L1409 0.96, 24 L1409 0.96, 10 L2048 0.96, 13 L4096 0.98)
    const int tiles = (L + 127) / 128, ctas = BH * (C::kParts + tiles);
    const bool one_each = DF == 32 && DV == 128 && BH * C::kParts <= kSMs && ctas > kSMs + 8 * ((tiles < 14 ? tiles : 14) - 2) &&
                          ctas <= 330 + 4 * tiles;
    const cudaError_t e =
        launch_ex(generic_state_tc_kernel<DF, DV>, dim3(C::kParts, BH), dim3(kThreadsS), C::kSmem, 1, !one_each, stream, tv, p);
    note_launch();
    const based_status st = check_launch("generic_state_tc_kernel");
    return e == cudaSuccess ? st : BASED_ERR_CUDA;
}
}  // namespace

based_status launch_state_generic_tc(const void* k, const void* v, float* kv, float* z, int BH, int L, int d_feat,
                                     int d_v, int cont, cudaStream_t stream) {
    auto go = [&](auto df_tag) {
        constexpr int DF = decltype(df_tag)::value;
        return d_v == 64 ? launch_state<DF, 64>(k, v, kv, z, BH, L, 64, cont, stream)
                         : launch_state<DF, 128>(k, v, kv, z, BH, L, d_v, cont, stream);         // 112 or 128
    };
    return d_feat == 8 ? go(std::integral_constant<int, 8>{})
                       : d_feat == 24 ? go(std::integral_constant<int, 24>{}) : go(std::integral_constant<int, 32>{});
}

}  // namespace based
