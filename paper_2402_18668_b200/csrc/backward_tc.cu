// based_prefill_backward, bf16 tensor-core path (tcgen05 / TMEM / TMA): the same three passes as
// the fp32 path (row statistics, dq, dk + dv; see backward_f32.cu for the formulas), with every
// 128 x 128 tile of (query, key) pairs evaluated by tensor-core products:
//
//   S  = Q_i K_j^T          (K = 16)          GV = G_i V_j^T   (K = d_v; G = dout, exact in bf16)
//   dq:   DS = (GV / D_i + b_i)(1/4 + S/16) [j<=i]  as bf16 in tensor memory,   dQ_i += DS K_j
//   dk/dv: the transposed products S^T = K_j Q_i^T, GV^T = V_j G_i^T;  W'^T = w(S^T) / D_i and DS^T in
//          tensor memory (over the scores, in place);   dV_j += W'^T G_i,   dK_j += DS^T Q_i
// 1/D_i is applied to the fp32 products, not to the operand: a = dout / D rounded to bf16 would
// break the near-cancellation of a_i.v_j + b_i for short prefixes.
//
// When the caller passes the forward output, statistics and dq take one sweep (a fifth mode):
//   dq_i = X_i / D_i + (m_i / D_i + b_i) Y_i,   X_i = sum_j w'_ij (gv_ij - m_i) k_j,   Y_i = sum_j w'_ij k_j
// holds for any m_i and needs neither D_i nor b_i while the keys are swept: D_i and E_i accumulate in
// registers, X and Y by MMA from two packed bf16 tiles, and 1/D_i, b_i, dq_i are formed in fp32 at the
// end.  m_i = dout_i . out_i is the weighted mean E_i / D_i of the gv_ij up to the rounding of out, so
// the packed products are as small as ds above and the part of dq that cancels against b_i stays in
// fp32 (without a centre the two separately rounded tiles would have to cancel).
//
// One CTA per (head, 128-row tile), 160 threads: warps 0-3 own one accumulator row each (the
// polynomial, masks and bf16 packing), warp 4 issues TMA loads and MMAs (converged, one elected lane).  The loop over
// the other side's tiles is sequential per CTA (loads of the next tile are in flight during the
// current one); parallelism comes from the (tile, head) grid.  q and k tiles are loaded 32
// columns wide (columns 16..31 are zero-filled by TMA) so that they serve both as K-major
// operands of the scores and as MN-major B operands of dQ / dK.  The work is O(L^2) per head, as
// in the fp32 path.  A fourth mode of the same kernel evaluates the forward pass in this form
// (scores, weights as bf16 in tensor memory, Y += P V, row sums): the tensor-core path of the
// feature dimensions 8, 24 and 32, which the chunked d' = 16 kernel does not cover.  All modes take
// d' (8, 16, 24, 32) as a parameter: the polynomial's coefficients 1/sqrt(d'), 1/(2 d'), a second K
// step of the scores above 16, and up to 32 gradient columns of dq and dk.
//
// Block-wise path (template flag XB; d' = 16, statistics in one sweep): linear in L.  The loops of the merged
// statistics + dq pass and of the dk/dv pass stop at the edges of the own tile's block of W tokens; all earlier
// blocks reach a query, and all later blocks a key, through one state tile each (block_state_tc.cu writes them:
// S = sum mono(k) v^T with row sums z for the queries, R = sum mono(q) (dout / D)^T with row sums R_b = sum b mono(q)
// for the keys, in the basis of the 153 distinct monomials of the feature map).  Before its loop such a CTA
// multiplies its own wide tile with the state tile (T = G S^T or V R^T, 128 x 160 in tensor memory), every row
// thread contracts its row of T with the monomials and the Jacobian of its q or k row, and the results start the
// accumulators that the loop's products add to; the dk/dv pass also writes the monomials of its k rows back to
// tensor memory as the A operand of dV = mono(K) R.
#include <math.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "sm100.cuh"

namespace based {
using namespace sm100;

namespace {
constexpr int kTile = 128;
constexpr int kThreadsB = 160;
constexpr int kModeStats = 0, kModeDq = 1, kModeDkDv = 2, kModeFwd = 3, kModeDqS = 4;
// the forward with the rounded weights' sums, for one chunk of d' 16, which gives the bits of prefill_tc_kernel's ROUNDED
constexpr int kModeFwdRounded = 5;
__host__ __device__ constexpr int base_mode(int mode) { return mode == kModeFwdRounded ? kModeFwd : mode; }
constexpr uint32_t kQKTile = kTile * 64;                 // [128][32] bf16, 64-byte rows, SWIZZLE_64B

// LT: rows of the tiles the CTA loops over (columns of the accumulators): 64 where that lets two CTAs
// share an SM (256 tensor-memory columns each), so that one CTA's row-thread pass overlaps the
// other's MMA bursts; 128 for the dk/dv pass at d_v 128, whose accumulators need more columns.
template <int DV, int MODE, int LT, bool XB = false> struct BCfg {
    static constexpr int kVB = (DV + 63) / 64;           // 64-column blocks of a [rows][DV] tile (112 -> 2, second partly zero)
    static constexpr uint32_t kWide = kVB * kTile * 128; // own tile: [128][64 * kVB] bf16 in SWIZZLE_128B blocks
    static constexpr uint32_t kNarrowL = LT * 64, kWideL = kVB * LT * 128;       // looped tiles
    // shared memory: resident narrow + wide tile, stages of (narrow + wide), (1/D, b) of two stages, barriers
    static constexpr uint32_t offResN = 0, offResW = offResN + kQKTile;
    // The next tile's scores are issued as soon as this tile's are read, where tensor memory holds the packed tiles beside the
    // scores: B2 H16 L1000 d_v 128 46.5 -> 44.5 us, B1 H8 L300 d_v 64 16.8 -> 16.3 per backward call.  Not where it takes
    // looped tiles of 32 rows (dk/dv at d_v 64: 31 -> 35 at B2 H8 L700, the own tile is read from shared memory twice as often)
    // or of 64 for 128 (dk/dv at d_v 128: 44 -> 54), and not where loops are two to four tiles (block-wise: no gain).
    static constexpr bool kEarly = !XB && MODE != kModeFwd && MODE != kModeDkDv;
    static constexpr int kNSt = kEarly ? 3 : 2;          // stages
    static constexpr uint32_t offStage = offResW + kWide, kStage = kNarrowL + kWideL;
    // a block state, transposed: [64 * kVB value columns][160 features] bf16 in five SWIZZLE_64B blocks of 32 features
    // (block-wise path); it lies from the second stage on, so that the first looped tile loads beside it
    static constexpr uint32_t kStateBlk = kVB * 64 * 64;
    static constexpr uint32_t kStateTile = 5 * kStateBlk;
    static constexpr uint32_t kStageArea = (XB && kStage + kStateTile > kNSt * kStage) ? kStage + kStateTile : kNSt * kStage;
    static constexpr uint32_t offB = offStage + kStageArea;
    static constexpr uint32_t offMisc = offB + 2 * LT * 8;
    static constexpr uint32_t kSmem = offMisc + 2048 + 1024;                    // barriers, the block state's row sums (160 floats), m (128)

    // tensor memory columns: scores, dout.v products, ds (dq pass; the dk/dv pass packs in place), accumulators
    static constexpr uint32_t colS = 0, colG = LT, colD = MODE == kModeFwd ? 0 : 2 * LT;    // forward: no dout.v product, the weights over the scores
    static constexpr uint32_t colD2 = colD + LT / 2;                                      // second packed tile (merged pass)
    static constexpr uint32_t colAcc = MODE == kModeDq ? 2 * LT + LT / 2                  // dQ (32)
                                       : MODE == kModeDqS ? 3 * LT                        // X (32), then Y (32)
                                       : MODE == kModeFwd ? LT                            // Y (64 * kVB)
                                                          : (LT == 32 ? 96 : 2 * LT < 160 ? 160 : 2 * LT);  // dV (64 * kVB): above the block
                                       // product (160 columns), or with 32-row looped tiles above its packed monomials (80): the
                                       // product is read before the first dV product is issued
    static constexpr uint32_t colAcc2 = colAcc + 32;                                      // merged pass: Y
    static constexpr uint32_t colK = colAcc + 64 * kVB;                                   // dK (32), dk/dv pass
    static constexpr uint32_t kColsUsed = MODE == kModeStats ? 2 * LT
                                          : MODE == kModeDq ? colAcc + 32
                                          : MODE == kModeDqS ? colAcc2 + 32
                                          : MODE == kModeFwd ? colAcc + 64 * kVB
                                                             : colK + 32;
    static constexpr uint32_t kCols = kColsUsed <= 128 ? 128 : kColsUsed <= 256 ? 256 : 512;
    static_assert(kColsUsed <= 512, "tensor memory budget");
};
enum { bRes = 0, bFull0, bFull1, bFull2, bMma, bRead, bAlu, bAcc, bFinal, bXs, bX0, bX1, bNum };

struct BParams {
    const __nv_bfloat16* o_raw;  // the forward output as a plain pointer [BH, L, dvw] (merged pass)
    const float2* stats_in;      // (1/D, b) per row (dq, dk/dv passes)
    float2* stats_out;           // statistics pass
    __nv_bfloat16* dq;           // [BH, L, 16]
    __nv_bfloat16* dk;
    unsigned int* err;
    int L, dvw, numerator_only;  // dvw: value head dimension of the caller's tensors (64, 112, 128)
    int df, kdim;                // feature dimension d', and d' rounded up to 16 (K extent of the scores)
    float s1, s2;                // w = 1 + s * s1 + s^2 * s2 (1 / sqrt d', 1 / (2 d'))
    // block-wise path: pairs inside a block of W tokens by tiles, the other blocks through their summed state
    int W, nblk;
    int heads, by_length;        // by_length: the longest loops of all heads first, else head by head
    int dout_H;                  // heads per sequence where dout lies [B, L, H, d_v]; else 0
    int overlapped;              // forward: this grid runs beside the one before it, and ends after it
    const float* sv;             // [BH x nblk][160]: row sums of the block states (z, or the b-weighted sums of phi(q))
};

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t*>(&v);
}
// AND of a predicate over the 128 row threads (named barrier 1): all of them get the same answer, so
// they leave their loop together and the warp-collective tensor-memory accesses stay converged; it
// also orders their shared-memory writes before the reads that follow
__device__ __forceinline__ bool rows_all(bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, 128, p;\n\t"
        "selp.b32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)pred)
        : "memory");
    return r != 0;
}
// pairs of fp32 values in one register pair
__device__ __forceinline__ uint64_t f32x2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void split_f32x2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul_f32x2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// Block-wise path, one row thread: T (160 fp32 columns of tensor memory, from column 0) holds the product of the
// row's wide operand with a block state in the monomial basis of block_state_tc_kernel
// (f < 16: x_f | 16 + 16 o + m: x_m x_(m+o) | 144 + m: x_m x_(m+8) | 152: 1), sv the state's row sums.
//   query row (merged statistics + dq pass): T_f = (S g_i)_f, sv = z:
//     den += mono(q_i) . z,  en += mono(q_i) . T,  gx = J^T (T - m_i z),  gy = J^T z      (J = d mono / d q_i)
//   key row (dk/dv pass): T_f = (R v_j)_f, sv = R_b:  gx = J^T (T + R_b); the monomials of k_j go back to tensor
//     memory as packed bf16 (80 columns from column 0, over the columns already read): the A operand of dV += mono(K) R
// Two features per instruction: f, f + 1 (f even) are x_m x_n and x_(m+1) x_(n+1), m even; where n is odd the pair's second
// factors and the sums that go to them lie across two words, in arrays of their own (xo; gxo, gyo).
template <bool KEYS>
__device__ __forceinline__ void block_rows(uint32_t tb, uint32_t lane_base, const float (&x)[16], const float* sv,
                                           float m_own, float& den, float& en, float (&gx)[16], float (&gy)[16]) {
    uint64_t xe[8], xo[8], gxe[8], gxo[8], gye[8], gyo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        xe[i] = f32x2(x[2 * i], x[2 * i + 1]);
        xo[i] = f32x2(x[2 * i + 1], x[(2 * i + 2) & 15]);
        gxe[i] = gxo[i] = gye[i] = gyo[i] = 0;
    }
    const uint64_t negm = f32x2(-m_own, -m_own);
    uint64_t den2 = f32x2(den, 0.f), en2 = f32x2(en, 0.f);
#pragma unroll
    for (int blk = 0; blk < 5; ++blk) {
        uint32_t tr[32], pk[16];
        tmem_ld32(tmem_addr(tb, lane_base, blk * 32), tr);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int f = blk * 32 + 2 * i;
            const int m = f < 16 ? f : f < 144 ? ((f - 16) & 15) : f - 144;
            const int n = f < 16 ? -1 : f < 144 ? ((m + ((f - 16) >> 4)) & 15) : m + 8;
            if (KEYS) pk[i] = 0u;
            if (f > 152) continue;
            const ulonglong2 z4 = *reinterpret_cast<const ulonglong2*>(sv + (f & ~3));       // broadcast: four row sums
            const uint64_t z = f & 2 ? z4.y : z4.x;
            const uint64_t a = f32x2(__uint_as_float(tr[2 * i]), __uint_as_float(tr[2 * i + 1]));
            if (f == 152) {                                  // the constant
                float z0, z1;
                split_f32x2(z, z0, z1);
                if (KEYS) pk[i] = pack_bf16x2(1.0f, 0.f);
                else {
                    den2 = add_f32x2(den2, f32x2(z0, 0.f));
                    en2 = add_f32x2(en2, f32x2(__uint_as_float(tr[2 * i]), 0.f));
                }
                continue;
            }
            const uint64_t xm = xe[m / 2], xn = n < 0 ? 0 : n & 1 ? xo[n / 2] : xe[n / 2];
            const uint64_t mono = n < 0 ? xm : mul_f32x2(xm, xn);
            const uint64_t bq = KEYS ? add_f32x2(a, z) : fma_f32x2(negm, z, a);
            if (KEYS) {
                float lo, hi;
                split_f32x2(mono, lo, hi);
                pk[i] = pack_bf16x2(lo, hi);
            } else {
                den2 = fma_f32x2(mono, z, den2);
                en2 = fma_f32x2(mono, a, en2);
            }
            uint64_t& gm = gxe[m / 2];
            uint64_t& hm = gye[m / 2];
            if (n < 0) {
                gm = add_f32x2(gm, bq);
                if (!KEYS) hm = add_f32x2(hm, z);
            } else {                                         // (m = n: both terms)
                uint64_t& gn = n & 1 ? gxo[n / 2] : gxe[n / 2];
                uint64_t& hn = n & 1 ? gyo[n / 2] : gye[n / 2];
                gm = fma_f32x2(xn, bq, gm);
                gn = fma_f32x2(xm, bq, gn);
                if (!KEYS) {
                    hm = fma_f32x2(xn, z, hm);
                    hn = fma_f32x2(xm, z, hn);
                }
            }
        }
        if (KEYS) tmem_st16(tmem_addr(tb, lane_base, blk * 16), pk);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        float a, b, c, d;
        split_f32x2(gxe[i], a, b);
        split_f32x2(gxo[(i + 7) & 7], c, d);                 // .. 2 i - 1, 2 i
        gx[2 * i] = a + d;
        split_f32x2(gxo[i], c, d);
        gx[2 * i + 1] = b + c;
        split_f32x2(gye[i], a, b);
        split_f32x2(gyo[(i + 7) & 7], c, d);
        gy[2 * i] = a + d;
        split_f32x2(gyo[i], c, d);
        gy[2 * i + 1] = b + c;
    }
    float a, b;
    split_f32x2(den2, a, b);
    den = a + b;
    split_f32x2(en2, a, b);
    en = a + b;
}
}  // namespace

// tm_n0 / tm_w0: narrow (q or k) and wide (a/g or v) tensor of the CTA's own (resident) tile;
// tm_n1 / tm_w1: of the tiles it loops over.
// XB: the block-wise path (merged statistics + dq pass and dk/dv pass, d' = 16); tm_st: the block states,
// transposed: [BH x nblk][d_v][160] bf16.  tm_out: the wide output (dv, or the forward output), stored by TMA.
template <int DV, int KIND, int LT, bool XB>
__global__ void __launch_bounds__(kThreadsB, base_mode(KIND) == kModeFwd ? 4 : 2)
    backward_tc_kernel(const __grid_constant__ CUtensorMap tm_n0, const __grid_constant__ CUtensorMap tm_w0,
                       const __grid_constant__ CUtensorMap tm_n1, const __grid_constant__ CUtensorMap tm_w1,
                       const __grid_constant__ CUtensorMap tm_st, const __grid_constant__ CUtensorMap tm_out,
                       const BParams p) {
    constexpr int MODE = base_mode(KIND);
    static_assert(!XB || MODE == kModeDqS || MODE == kModeDkDv, "block-wise path: the two passes that use it");
    static_assert(MODE != kModeFwd || (DV == 64 && LT == 64), "the forward: d_v 64");
    using C = BCfg<DV, MODE, LT, XB>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::offMisc);
    uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(bars + bNum);
    volatile uint32_t* abort_flag = tmem_base_s + 1;
    float* s_b = reinterpret_cast<float*>(smem + C::offB);
    float* s_sv = reinterpret_cast<float*>(smem + C::offMisc + 256);
    float* s_m = reinterpret_cast<float*>(smem + C::offMisc + 1024);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ntiles = (p.L + kTile - 1) / kTile;
    // own tile: the longest loops first (dq, statistics: last query tiles; dk/dv: first key tiles)
    int turn = p.by_length ? blockIdx.x / p.heads : blockIdx.x % ntiles;
    int head = p.by_length ? blockIdx.x - turn * p.heads : blockIdx.x / ntiles;
    if (XB) {
        // First the tiles that need no block state, all heads': they run beside the states' kernel, on what it leaves of the chip
        // (us per backward call, after it / beside it: B4 H16 L2048 d_v64 96.2 / 93.0, d_v128 130.1 / 124.5, L4096 245.4 / 238.4, B8 H16
        // L1024 d_v64 87.1 / 85.7, B4 H8 L2048 67.2 / 66.5; the states' kernel held to the registers that leave room for one of these
        // CTAs on its own SMs too, at d_v 64: 95.0)
        const int alone = MODE == kModeDkDv ? ntiles - (p.nblk - 1) * (p.W / kTile) : p.W / kTile, rest = ntiles - alone;
        const int i = (int)blockIdx.x - p.heads * alone;
        head = i < 0 ? blockIdx.x / alone : i / rest;
        turn = i < 0 ? rest + blockIdx.x % alone : i % rest;
    }
    const int own = MODE == kModeDkDv ? turn : ntiles - 1 - turn;
    const int r0 = own * kTile;
    // looped tiles (LT rows each): keys 0 .. end of the own tile, or queries from the own tile's first row on
    // block-wise path: the loop stays inside the own tile's block of W tokens; the blocks before it (queries) or
    // after it (keys) enter through their summed state, if there are any (cross)
    const int blk = XB ? r0 / p.W : 0;
    const bool cross = XB && (MODE == kModeDkDv ? blk + 1 < p.nblk : blk > 0);
    const int first = MODE == kModeDkDv ? r0 / LT : (XB ? blk * p.W / LT : 0);
    const int last = MODE == kModeDkDv ? (min(p.L, XB ? (blk + 1) * p.W : p.L) - 1) / LT : (min(p.L, r0 + kTile) - 1) / LT;
    const int nloop = last - first + 1;

    if (tid == 0) {
        mbar_init(&bars[bRes], 1); mbar_init(&bars[bFull0], 1); mbar_init(&bars[bFull1], 1); mbar_init(&bars[bFull2], 1);
        mbar_init(&bars[bMma], 1); mbar_init(&bars[bRead], 128); mbar_init(&bars[bAlu], 128);
        mbar_init(&bars[bAcc], 1); mbar_init(&bars[bFinal], 1);
        mbar_init(&bars[bXs], 1); mbar_init(&bars[bX0], 1); mbar_init(&bars[bX1], 128);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 4) { tmem_alloc(tmem_base_s, C::kCols); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = *tmem_base_s;
    bool ok = true;
    // A dependent launch: set up while the grid ahead drains.  Behind a kernel of states, which has waited for everything before it,
    // the forward and the tiles that need no state start at once.
    if (MODE == kModeFwd ? !p.overlapped : !XB || cross) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    // descriptors: narrow tiles (64-byte rows, SWIZZLE_64B), wide tiles (128-byte rows, SWIZZLE_128B, 64-column blocks)
    constexpr uint64_t dN = make_smem_desc_base(16, 512, kSwizzle64B);                  // K-major, or MN-major one block
    constexpr uint64_t dW = make_smem_desc_base(kTile * 128, 1024, kSwizzle128B);       // own wide tile (128 rows per block)
    constexpr uint64_t dWL = make_smem_desc_base(LT * 128, 1024, kSwizzle128B);         // looped wide tile (LT rows per block)
    constexpr uint32_t iS = make_idesc_bf16(128, LT, 0, 0);                             // both operands K-major
    constexpr uint32_t iN32 = make_idesc_bf16(128, 32, 0, 1);                           // A from TMEM, B MN-major narrow
    constexpr uint32_t iNV = make_idesc_bf16(128, 64 * C::kVB, 0, 1);                   // A from TMEM, B MN-major wide
    constexpr uint64_t dStN = make_smem_desc_base(C::kStateBlk, 512, kSwizzle64B);      // block state as B over d_v: MN-major
    constexpr uint32_t iT = make_idesc_bf16(128, 160, 0, 1);                            // own wide x state^T
    constexpr uint32_t iXV = make_idesc_bf16(128, 64 * C::kVB, 0, 0);                   // A from TMEM, B K-major: the state over features

    if (warp == 4) {
        {
            // the whole warp runs this block; one elected lane issues the MMAs, commits and loads (see mma_ss_w)
            const uint32_t lead = elect_one();
            const int gb = p.dout_H ? head / p.dout_H : 0, gh = head - gb * p.dout_H;      // the head in the coordinates of a dout [B][L][H][d_v]
            const uint32_t aResN = smem_u32(smem + C::offResN), aResW = smem_u32(smem + C::offResW);
            auto load_stage = [&](int it) {
                if (!lead || it >= nloop) return;
                const int s = it % C::kNSt;
                uint8_t* st = smem + C::offStage + s * C::kStage;
                const int row = (first + it) * LT;
                mbar_arrive_expect_tx(&bars[bFull0 + s], C::kStage);
                tma_load_3d(st, &tm_n1, &bars[bFull0 + s], 0, row, head);
#pragma unroll
                for (int b = 0; b < C::kVB; ++b)
                    if (MODE == kModeDkDv && p.dout_H) tma_load_4d(st + C::kNarrowL + b * (LT * 128), &tm_w1, &bars[bFull0 + s], b * 64, gh, row, gb);
                    else tma_load_3d(st + C::kNarrowL + b * (LT * 128), &tm_w1, &bars[bFull0 + s], b * 64, row, head);
            };
            if (lead) {
            mbar_arrive_expect_tx(&bars[bRes], MODE == kModeFwd ? kQKTile : kQKTile + C::kWide);
            tma_load_3d(smem + C::offResN, &tm_n0, &bars[bRes], 0, r0, head);
            if (MODE != kModeFwd) {
#pragma unroll
                for (int b = 0; b < C::kVB; ++b)
                    if (MODE != kModeDkDv && p.dout_H) tma_load_4d(smem + C::offResW + b * (kTile * 128), &tm_w0, &bars[bRes], b * 64, gh, r0, gb);
                    else tma_load_3d(smem + C::offResW + b * (kTile * 128), &tm_w0, &bars[bRes], b * 64, r0, head);
            }
            if (cross) {
                mbar_arrive_expect_tx(&bars[bXs], C::kStateTile);
#pragma unroll
                for (int b = 0; b < 5; ++b)
                    tma_load_3d(smem + C::offStage + C::kStage + b * C::kStateBlk, &tm_st, &bars[bXs], b * 32, 0,
                                head * p.nblk + blk);
            }
            }
            for (int i = 0; i < (cross ? 1 : C::kNSt); ++i) load_stage(i);     // (the block state lies over the others)
            ok = mbar_wait(&bars[bRes], 0, abort_flag);
            if (cross && ok) {
                const uint32_t aSt = smem_u32(smem + C::offStage + C::kStage);
                ok = mbar_wait(&bars[bXs], 0, abort_flag);
                tc_fence_after();
                // T = own wide tile x state^T (K = d_v), 160 columns from column 0
#pragma unroll
                for (int kk = 0; kk < DV / 16; ++kk) {
                    const uint32_t off = ((kk >> 2) * (kTile * 128) + (kk & 3) * 32) >> 4;
                    const uint32_t offS = (kk * 1024) >> 4;        // sixteen value columns = sixteen 64-byte rows of every block
                    if (kk == 0)
                        mma_ss_w<false>(lead, tb, desc_lo(dW) + (aResW >> 4) + off, desc_hi(dW), desc_lo(dStN) + (aSt >> 4) + offS,
                                         desc_hi(dStN), iT);
                    else
                        mma_ss_w<true>(lead, tb, desc_lo(dW) + (aResW >> 4) + off, desc_hi(dW), desc_lo(dStN) + (aSt >> 4) + offS,
                                        desc_hi(dStN), iT);
                }
                mma_commit_w(lead, &bars[bX0]);
                if (MODE == kModeDkDv) {
                    // dV = mono(K) (tensor memory, written by the row threads) x state (K-major: 64-byte rows of 32
                    // features, 160 = 10 K-steps of 32 bytes)
                    if (ok) ok = mbar_wait(&bars[bX1], 0, abort_flag);
                    tc_fence_after();
                    if (ok) {
#pragma unroll
                        for (int k = 0; k < 10; ++k) {
                            const uint32_t offK = ((k >> 1) * C::kStateBlk + (k & 1) * 32) >> 4;
                            if (k == 0)
                                mma_ts_w<false>(lead, tb + C::colAcc, tb + k * 8, desc_lo(dN) + (aSt >> 4) + offK, desc_hi(dN), iXV);
                            else
                                mma_ts_w<true>(lead, tb + C::colAcc, tb + k * 8, desc_lo(dN) + (aSt >> 4) + offK, desc_hi(dN), iXV);
                        }
                    }
                } else {
                    if (ok) ok = mbar_wait(&bars[bX1], 0, abort_flag);     // the rows have read T: the scores may overwrite it
                    tc_fence_after();
                }
            }
            // scores and dout.v products of a looped tile: rows = own tile, columns = looped tile
            auto scores = [&](int it) -> bool {
                const uint32_t aN = smem_u32(smem + C::offStage + (it % C::kNSt) * C::kStage), aW = aN + C::kNarrowL;
                if (!mbar_wait(&bars[bFull0 + it % C::kNSt], (it / C::kNSt) & 1, abort_flag)) return false;
                tc_fence_after();
                mma_ss_w<false>(lead, tb + C::colS, desc_lo(dN) + (aResN >> 4), desc_hi(dN), desc_lo(dN) + (aN >> 4),
                                 desc_hi(dN), iS);
                if (p.kdim > 16)                             // feature dimensions 24 and 32: second K-step
                    mma_ss_w<true>(lead, tb + C::colS, desc_lo(dN) + (aResN >> 4) + 2, desc_hi(dN), desc_lo(dN) + (aN >> 4) + 2,
                                    desc_hi(dN), iS);
                // own wide tile x looped wide tile^T over d_v
#pragma unroll
                for (int kk = 0; kk < (MODE == kModeFwd ? 0 : DV / 16); ++kk) {
                    const uint32_t off = ((kk >> 2) * (kTile * 128) + (kk & 3) * 32) >> 4;
                    const uint32_t offL = ((kk >> 2) * (LT * 128) + (kk & 3) * 32) >> 4;
                    if (kk == 0)
                        mma_ss_w<false>(lead, tb + C::colG, desc_lo(dW) + (aResW >> 4) + off, desc_hi(dW),
                                         desc_lo(dWL) + (aW >> 4) + offL, desc_hi(dWL), iS);
                    else
                        mma_ss_w<true>(lead, tb + C::colG, desc_lo(dW) + (aResW >> 4) + off, desc_hi(dW),
                                        desc_lo(dWL) + (aW >> 4) + offL, desc_hi(dWL), iS);
                }
                mma_commit_w(lead, &bars[bMma]);
                return true;
            };
            if (C::kEarly && ok) ok = scores(0);
            for (int it = 0; it < nloop && ok; ++it) {
                const int s = it % C::kNSt;
                const uint32_t aN = smem_u32(smem + C::offStage + s * C::kStage), aW = aN + C::kNarrowL;
                if (!C::kEarly) {
                    // once these products are done, so are the previous iteration's (in-order pipe): its stage is free, and
                    // after the first one's those that the block state lay over
                    ok = scores(it) && mbar_wait(&bars[bMma], it & 1, abort_flag);
                    if (!ok) break;
                    if (it > 0 || cross) load_stage(it + 1);
                } else {
                    // the rows have read this tile's scores: the next tile's are formed while they work on them
                    if (it + 1 < nloop) ok = mbar_wait(&bars[bRead], it & 1, abort_flag) && scores(it + 1);
                    // the stage of the tile before is free once its last products are done (statistics: its scores, which the
                    // rows have read)
                    if (it > 0 && ok) ok = MODE == kModeStats || mbar_wait(&bars[bAcc], (it - 1) & 1, abort_flag);
                    if (!ok) break;
                    if (it > 0) load_stage(it - 1 + C::kNSt);
                }
                if (MODE == kModeStats) continue;
                ok = mbar_wait(&bars[bAlu], it & 1, abort_flag);
                if (!ok) break;
                tc_fence_after();
                if (MODE == kModeDq) {
                    // dQ += DS (tensor memory, LT keys = LT/16 K-steps) x K_j (MN-major, 32 columns)
#pragma unroll
                    for (int k = 0; k < LT / 16; ++k) {
                        if (it == 0 && k == 0)
                            mma_ts_w<false>(lead, tb + C::colAcc, tb + C::colD + k * 8, desc_lo(dN) + ((aN + k * 1024) >> 4),
                                             desc_hi(dN), iN32);
                        else
                            mma_ts_w<true>(lead, tb + C::colAcc, tb + C::colD + k * 8, desc_lo(dN) + ((aN + k * 1024) >> 4),
                                            desc_hi(dN), iN32);
                    }
                } else if (MODE == kModeDqS) {
                    // X += (w' (gv - m)) K_j and Y += w' K_j: two packed tiles in tensor memory, the same B operand
#pragma unroll
                    for (int k = 0; k < LT / 16; ++k) {
                        if (it == 0 && k == 0 && !cross) {
                            mma_ts_w<false>(lead, tb + C::colAcc, tb + C::colD + k * 8, desc_lo(dN) + ((aN + k * 1024) >> 4),
                                             desc_hi(dN), iN32);
                            mma_ts_w<false>(lead, tb + C::colAcc2, tb + C::colD2 + k * 8, desc_lo(dN) + ((aN + k * 1024) >> 4),
                                             desc_hi(dN), iN32);
                        } else {
                            mma_ts_w<true>(lead, tb + C::colAcc, tb + C::colD + k * 8, desc_lo(dN) + ((aN + k * 1024) >> 4),
                                            desc_hi(dN), iN32);
                            mma_ts_w<true>(lead, tb + C::colAcc2, tb + C::colD2 + k * 8, desc_lo(dN) + ((aN + k * 1024) >> 4),
                                            desc_hi(dN), iN32);
                        }
                    }
                } else if (MODE == kModeFwd) {
                    // Y += P (tensor memory) x V_j
#pragma unroll
                    for (int k = 0; k < LT / 16; ++k) {
                        if (it == 0 && k == 0)
                            mma_ts_w<false>(lead, tb + C::colAcc, tb + C::colD + k * 8, desc_lo(dWL) + ((aW + k * 2048) >> 4),
                                             desc_hi(dWL), iNV);
                        else
                            mma_ts_w<true>(lead, tb + C::colAcc, tb + C::colD + k * 8, desc_lo(dWL) + ((aW + k * 2048) >> 4),
                                            desc_hi(dWL), iNV);
                    }
                } else if (MODE == kModeDkDv) {
                    // dV += W'^T (over the scores) x G_i;  dK += DS^T (over GV) x Q_i
#pragma unroll
                    for (int k = 0; k < LT / 16; ++k) {
                        if (it == 0 && k == 0 && !cross) {
                            mma_ts_w<false>(lead, tb + C::colAcc, tb + C::colS + k * 8, desc_lo(dWL) + ((aW + k * 2048) >> 4),
                                             desc_hi(dWL), iNV);
                            mma_ts_w<false>(lead, tb + C::colK, tb + C::colG + k * 8, desc_lo(dN) + ((aN + k * 1024) >> 4),
                                             desc_hi(dN), iN32);
                        } else {
                            mma_ts_w<true>(lead, tb + C::colAcc, tb + C::colS + k * 8, desc_lo(dWL) + ((aW + k * 2048) >> 4),
                                            desc_hi(dWL), iNV);
                            mma_ts_w<true>(lead, tb + C::colK, tb + C::colG + k * 8, desc_lo(dN) + ((aN + k * 1024) >> 4),
                                            desc_hi(dN), iN32);
                        }
                    }
                }
                if (C::kEarly) mma_commit_w(lead, &bars[bAcc]);
            }
            if (ok) mma_commit_w(lead, &bars[bFinal]);
        }
    } else {
        // ===================================================================== row threads
        const int t = tid;                                   // accumulator row == TMEM lane
        const uint32_t lane_base = (uint32_t)warp * 32u;
        const int row = r0 + t;                              // query (statistics, dq) or key (dk/dv) of this thread
        float den = 0.f, en = 0.f;
        float2 st_own = make_float2(0.f, 0.f);               // (1/D, b) of this thread's query (dq pass)
        if (MODE == kModeDq && row < p.L) st_own = p.stats_in[(size_t)head * p.L + row];
        // merged pass: the products dout_i . v_j enter the packed tile relative to m_i = dout_i . out_i, which
        // is their weighted mean E_i / D_i up to the rounding of out: the part of dq that cancels against
        // b_i is then formed in fp32 at the end, not from two separately rounded bf16 tiles
        // the block state's row sums: read by the row threads only, after their next barrier
        if (XB && cross) {
            const float* svp = p.sv + ((size_t)head * p.nblk + blk) * 160;
            s_sv[t] = svp[t];
            if (t < 32) s_sv[128 + t] = svp[128 + t];
        }
        float m_own = 0.f;
        if (MODE == kModeDqS && !p.numerator_only) {
            // a warp's 32 rows of out lie one after the other in global memory: every load instruction takes 512
            // consecutive bytes (two rows at d_v 128, four at d_v 64; 448, two rows, at d_v 112, where a thread per row had
            // read 14 pieces of out and dout each: 512 -> 462 us per backward call at B8 H16 L4096); the matching piece of dout comes from the own
            // tile in shared memory, and the lanes of a row add up their parts
            constexpr int PPR = DV / 8;                       // 16-byte pieces per row
            constexpr int NI = PPR;                           // load instructions per warp: 32 rows x PPR pieces / 32 lanes
            const int wrow0 = r0 + warp * 32;
            const uint4* op = reinterpret_cast<const uint4*>(p.o_raw + ((size_t)head * p.L + wrow0) * p.dvw);
            const int np = DV == 64 ? PPR : p.dvw / 8;        // pieces of a row in memory
            uint4 ob[NI];
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const int pc = i * 32 + lane, rr = pc / PPR, c = pc % PPR;  // piece of the warp's 32 x PPR
                ob[i] = wrow0 + rr < p.L && c < np ? op[rr * np + c] : make_uint4(0u, 0u, 0u, 0u);
            }
            ok = rows_all(mbar_wait(&bars[bRes], 0, abort_flag));
#pragma unroll
            for (int i0 = 0; i0 < NI; i0 += 8) {
                float d[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int pc = (i0 + i) * 32 + lane;
                    const int rr = warp * 32 + pc / PPR, c = pc % PPR;       // row of the tile, piece of the row
                    const uint4 u = *reinterpret_cast<const uint4*>(smem + C::offResW + (c >> 3) * (kTile * 128) + rr * 128 +
                                                                    (((c & 7) ^ (rr & 7)) << 4));
                    const __nv_bfloat162* ha = reinterpret_cast<const __nv_bfloat162*>(&u);
                    const __nv_bfloat162* hb = reinterpret_cast<const __nv_bfloat162*>(&ob[i0 + i]);
                    d[i] = 0.f;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 fa = __bfloat1622float2(ha[e]), fb = __bfloat1622float2(hb[e]);
                        d[i] = fmaf(fa.x, fb.x, d[i]);
                        d[i] = fmaf(fa.y, fb.y, d[i]);
                    }
                }
                // sums over the lanes of a row, eight rows at once: at every step a lane passes half of its values on and keeps
                // the other half, so that lane i is left with load i's row (7 or 8 exchanges for 24 or 32)
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) {
                    const bool up = lane & o;
#pragma unroll
                    for (int j = 0; j < o; ++j) {
                        const float give = up ? d[j] : d[j + o], keep = up ? d[j + o] : d[j];
                        d[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                    }
                }
                if (PPR == 16) d[0] += __shfl_xor_sync(0xffffffffu, d[0], 8);
                s_m[warp * 32 + ((i0 + (lane & 7)) * 32 + lane) / PPR] = d[0];
            }
            __syncwarp();
            m_own = s_m[t];
        }
        if (XB && cross) {
            // the blocks before (queries) or after (keys) the own one, through their summed state
            ok = rows_all(mbar_wait(&bars[bRes], 0, abort_flag) && mbar_wait(&bars[bX0], 0, abort_flag));
            tc_fence_after();
            if (ok) {
                // this thread's q or k row: 64-byte rows, SWIZZLE_64B (16-byte pieces 0 and 1)
                float x[16], gx[16], gy[16];
                const uint8_t* xrow = smem + C::offResN + t * 64;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const uint4 u = *reinterpret_cast<const uint4*>(xrow + ((c ^ ((t >> 1) & 3)) << 4));
                    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 fv = __bfloat1622float2(h[i]);
                        x[c * 8 + 2 * i] = fv.x;
                        x[c * 8 + 2 * i + 1] = fv.y;
                    }
                }
                block_rows<MODE == kModeDkDv>(tb, lane_base, x, s_sv, m_own, den, en, gx, gy);
                // the sums start the accumulators that the loop's products add to: X and Y, or dK
                uint32_t o[16], zero[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) { o[i] = __float_as_uint(gx[i]); zero[i] = 0u; }
                tmem_st16(tmem_addr(tb, lane_base, MODE == kModeDkDv ? C::colK : C::colAcc), o);
                tmem_st16(tmem_addr(tb, lane_base, (MODE == kModeDkDv ? C::colK : C::colAcc) + 16), zero);
                if (MODE == kModeDqS) {
#pragma unroll
                    for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(gy[i]);
                    tmem_st16(tmem_addr(tb, lane_base, C::colAcc2), o);
                    tmem_st16(tmem_addr(tb, lane_base, C::colAcc2 + 16), zero);
                }
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(&bars[bX1]);
            }
        }
        const uint64_t k1 = f32x2(p.s1, p.s1), k2 = f32x2(p.s2, p.s2), k22 = f32x2(2.0f * p.s2, 2.0f * p.s2), one = f32x2(1.f, 1.f);
        const uint64_t negm = f32x2(-m_own, -m_own), own_d = f32x2(st_own.x, st_own.x), own_b = f32x2(st_own.y, st_own.y);
        uint64_t den2 = f32x2(den, 0.f), en2 = f32x2(en, 0.f);
        // the packed tiles of 32 columns, in place of columns already read
        auto packed_out = [&](int blk, const uint32_t (&pw)[16], const uint32_t (&pd)[16]) {
            if (MODE == kModeDq || MODE == kModeDqS) tmem_st16(tmem_addr(tb, lane_base, C::colD + blk * 16), pd);
            if (MODE == kModeDqS) tmem_st16(tmem_addr(tb, lane_base, C::colD2 + blk * 16), pw);
            if (MODE == kModeFwd) tmem_st16(tmem_addr(tb, lane_base, C::colD + blk * 16), pw);
            if (MODE == kModeDkDv) {
                tmem_st16(tmem_addr(tb, lane_base, C::colS + blk * 16), pw);
                tmem_st16(tmem_addr(tb, lane_base, C::colG + blk * 16), pd);
            }
        };
        // after the tile's last tensor-memory load: the next tile's scores may overwrite these
        auto have_read = [&](int blk) {
            if (C::kEarly && blk == LT / 32 - 1) {
                tc_fence_before();
                mbar_arrive(&bars[bRead]);
            }
        };
        bool packed_ok = true;
        for (int it = 0; it < nloop && ok; ++it) {
            const int c0 = (first + it) * LT;                // first row of the looped tile (columns of the accumulators)
            if (MODE == kModeDkDv && t < LT) {               // 1/D and b of the looped queries
                const float2 st = c0 + t < p.L ? p.stats_in[(size_t)head * p.L + c0 + t] : make_float2(0.f, 0.f);
                s_b[(it & 1) * 2 * LT + t] = st.x;
                s_b[(it & 1) * 2 * LT + LT + t] = st.y;
            }
            ok = rows_all(packed_ok && mbar_wait(&bars[bMma], it & 1, abort_flag));
            if (!ok) break;
            tc_fence_after();
            // the packed tiles are free once the products of the tile before are done
            auto may_pack = [&]() {
                if (C::kEarly && MODE != kModeStats && it > 0) {
                    packed_ok = __all_sync(~0u, mbar_wait(&bars[bAcc], (it - 1) & 1, abort_flag)) && packed_ok;
                    tc_fence_after();
                }
            };
            // one pass over the tile's LT accumulator columns of this row, 32 at a time and two pairs per instruction.  The
            // warp's 32 rows meet 32 columns on one of three ways: all pairs live, none (zeros, nothing read), or some
            // (MASKED: on the diagonal or at the end of the sequence).
            auto pass = [&](auto masked_tag, int blk) {
                constexpr bool MASKED = decltype(masked_tag)::value;
                uint32_t sr[32], gr[32];
                // forward (d_v 64): the second sixteen columns are on their way while the first are worked on (38.3 -> 36.7 us at
                // B4 H16 L2048 d' 24; at d_v 128, and in the other passes, no gain or 1 to 2 % slower)
                constexpr bool kHalves = MODE == kModeFwd;
                uint32_t (&s0)[16] = *reinterpret_cast<uint32_t (*)[16]>(sr), (&s1)[16] = *reinterpret_cast<uint32_t (*)[16]>(sr + 16);
                if (kHalves) tmem_ld16(tmem_addr(tb, lane_base, C::colS + blk * 32), s0);
                else tmem_ld32(tmem_addr(tb, lane_base, C::colS + blk * 32), sr);
                if (MODE != kModeFwd) tmem_ld32(tmem_addr(tb, lane_base, C::colG + blk * 32), gr);
                tmem_wait_ld();
                if (kHalves) tmem_ld16(tmem_addr(tb, lane_base, C::colS + blk * 32 + 16), s1);
                have_read(blk);
                uint32_t pw[16], pd[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    if (kHalves && i == 8) tmem_wait_ld();
                    const uint64_t sv = f32x2(__uint_as_float(sr[2 * i]), __uint_as_float(sr[2 * i + 1]));
                    const uint64_t gv = MODE == kModeFwd ? 0 : f32x2(__uint_as_float(gr[2 * i]), __uint_as_float(gr[2 * i + 1]));
                    // pair (query, key): own row is the query except in the dk/dv pass
                    bool live0 = true, live1 = true;
                    if (MASKED) {
                        const int col = c0 + blk * 32 + 2 * i;
                        live0 = MODE == kModeDkDv ? (row <= col && col < p.L) : col <= row;
                        live1 = MODE == kModeDkDv ? (row <= col + 1 && col + 1 < p.L) : col + 1 <= row;
                    }
                    auto masked = [&](uint64_t v) {
                        if (!MASKED) return v;
                        float lo, hi;
                        split_f32x2(v, lo, hi);
                        return f32x2(live0 ? lo : 0.f, live1 ? hi : 0.f);
                    };
                    // w = 1 + s / sqrt(d') + s^2 / (2 d') and its derivative
                    uint64_t w = 0, dw = 0, ds = 0;
                    if (MODE != kModeDq) w = masked(fma_f32x2(sv, fma_f32x2(sv, k2, k1), one));
                    if (MODE == kModeDq || MODE == kModeDqS || MODE == kModeDkDv) dw = fma_f32x2(sv, k22, k1);
                    if (MODE == kModeDqS) dw = masked(dw);
                    if ((MODE == kModeFwd && KIND != kModeFwdRounded) || MODE == kModeStats || MODE == kModeDqS) den2 = add_f32x2(den2, w);
                    if (MODE == kModeStats || MODE == kModeDqS) en2 = fma_f32x2(w, gv, en2);
                    if (MODE == kModeDqS) {
                        ds = mul_f32x2(dw, add_f32x2(gv, negm));             // first tile: w' (gv - m); second: w'
                        w = dw;
                    }
                    // (masked by selection: 0 times a non-finite product would be NaN in pairs that do not count)
                    if (MODE == kModeDq) ds = masked(mul_f32x2(fma_f32x2(gv, own_d, own_b), dw));
                    if (MODE == kModeDkDv) {
                        const int c = (it & 1) * 2 * LT + blk * 32 + 2 * i;
                        const uint64_t qd = *reinterpret_cast<const uint64_t*>(s_b + c);
                        ds = masked(mul_f32x2(fma_f32x2(gv, qd, *reinterpret_cast<const uint64_t*>(s_b + LT + c)), dw));
                        w = mul_f32x2(w, qd);                // dv_j = sum_i (w_ij / D_i) G_i
                    }
                    float lo, hi;
                    split_f32x2(w, lo, hi);
                    pw[i] = pack_bf16x2(lo, hi);
                    if (KIND == kModeFwdRounded) den2 = add_f32x2(den2, f32x2(__uint_as_float(pw[i] << 16), __uint_as_float(pw[i] & 0xffff0000u)));
                    split_f32x2(ds, lo, hi);
                    pd[i] = pack_bf16x2(lo, hi);
                }
                if (blk == 0) may_pack();
                packed_out(blk, pw, pd);
            };
            if (MODE == kModeFwd && c0 + LT <= r0) {         // two column groups in flight (63 -> 60 us at B4 H16 L2048 d_v 128 when those ran here)
#pragma unroll
                for (int blk = 0; blk < LT / 32; ++blk) pass(std::false_type{}, blk);
            } else
#pragma unroll 1
            for (int blk = 0; blk < LT / 32; ++blk) {
                const int cb = c0 + blk * 32, rw = r0 + warp * 32;
                const bool dead = MODE == kModeDkDv ? cb < rw : cb > rw;
                const bool some = cb == rw || (MODE == kModeDkDv && cb + 32 > p.L);
                if (dead) {
                    uint32_t z[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) z[i] = 0u;
                    have_read(blk);
                    if (blk == 0) may_pack();
                    packed_out(blk, z, z);
                } else if (some) {
                    pass(std::true_type{}, blk);
                } else {
                    pass(std::false_type{}, blk);
                }
            }
            if (MODE != kModeStats) {
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(&bars[bAlu]);
            }
        }
        {
            float a, b;
            split_f32x2(den2, a, b);
            den = a + b;
            split_f32x2(en2, a, b);
            en = a + b;
        }
        if (MODE != kModeStats) ok = rows_all(ok && packed_ok && mbar_wait(&bars[bFinal], 0, abort_flag));
        tc_fence_after();
        // tcgen05.ld is a warp-collective: every lane takes part, only the stores depend on the row
        const bool store = ok && row < p.L;
        const size_t grow = (size_t)head * p.L + (store ? row : 0);
        if (MODE == kModeStats || MODE == kModeDqS) {
            const float dinv = p.numerator_only ? 1.0f : 1.0f / (den + kEps);
            const float bq = p.numerator_only ? 0.0f : -en * dinv * dinv;
            if (store) p.stats_out[grow] = make_float2(dinv, bq);
            if (MODE == kModeDqS && ok) {
                // dq_i = X_i / D_i + (m_i / D_i + b_i) Y_i
                const float cy = fmaf(m_own, dinv, bq);
                uint32_t rx[16], ry[16];
                for (int h = 0; h < (p.df + 15) / 16; ++h) {     // p.df is uniform: 8, 16, 24, 32 gradient columns
                    tmem_ld16(tmem_addr(tb, lane_base, C::colAcc + h * 16), rx);
                    tmem_ld16(tmem_addr(tb, lane_base, C::colAcc2 + h * 16), ry);
                    tmem_wait_ld();
                    if (store) {
                        uint32_t o[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            o[i] = pack_bf16x2(fmaf(__uint_as_float(rx[2 * i]), dinv, cy * __uint_as_float(ry[2 * i])),
                                               fmaf(__uint_as_float(rx[2 * i + 1]), dinv, cy * __uint_as_float(ry[2 * i + 1])));
                        uint4* dst = reinterpret_cast<uint4*>(p.dq + grow * p.df + h * 16);
                        dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
                        if (h * 16 + 8 < p.df) dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
                    }
                }
            }
        } else if (ok) {                                     // ok is uniform over the row threads (rows_all)
            // the d' gradient columns of dq (colAcc) or dk (colK), 16 at a time (p.df is uniform)
            for (int h = 0; h < (MODE == kModeFwd ? 0 : (p.df + 15) / 16); ++h) {
                uint32_t r[16];
                tmem_ld16(tmem_addr(tb, lane_base, (MODE == kModeDq ? C::colAcc : C::colK) + h * 16), r);
                tmem_wait_ld();
                if (store) {
                    uint4 o0, o1;
                    o0.x = pack_bf16x2(__uint_as_float(r[0]), __uint_as_float(r[1]));
                    o0.y = pack_bf16x2(__uint_as_float(r[2]), __uint_as_float(r[3]));
                    o0.z = pack_bf16x2(__uint_as_float(r[4]), __uint_as_float(r[5]));
                    o0.w = pack_bf16x2(__uint_as_float(r[6]), __uint_as_float(r[7]));
                    o1.x = pack_bf16x2(__uint_as_float(r[8]), __uint_as_float(r[9]));
                    o1.y = pack_bf16x2(__uint_as_float(r[10]), __uint_as_float(r[11]));
                    o1.z = pack_bf16x2(__uint_as_float(r[12]), __uint_as_float(r[13]));
                    o1.w = pack_bf16x2(__uint_as_float(r[14]), __uint_as_float(r[15]));
                    uint4* dst = reinterpret_cast<uint4*>((MODE == kModeDq ? p.dq : p.dk) + grow * p.df + h * 16);
                    dst[0] = o0;
                    if (h * 16 + 8 < p.df) dst[1] = o1;
                }
            }
            if (MODE == kModeDkDv || MODE == kModeFwd) {
                // the wide accumulator row: dv, or the forward output scaled by 1 / (denominator + eps)
                // through the own wide tile's place in shared memory (its products are done) in the layout of a TMA box,
                // [128 rows][64 columns] blocks with 128-byte rows, SWIZZLE_128B, and out by TMA: whole 128-byte lines
                // per row where a store per row thread would touch 32 rows per instruction.  Rows and columns past the
                // tensor's end are clipped by the store.
                const float sc = (MODE == kModeFwd && !p.numerator_only) ? 1.0f / (den + kEps) : 1.0f;
                for (int c = 0; c < p.dvw / 16; ++c) {       // p.dvw is uniform
                    uint32_t rv[16];
                    tmem_ld16(tmem_addr(tb, lane_base, C::colAcc + c * 16), rv);
                    tmem_wait_ld();
                    uint4 a, b;
                    a.x = pack_bf16x2(__uint_as_float(rv[0]) * sc, __uint_as_float(rv[1]) * sc);
                    a.y = pack_bf16x2(__uint_as_float(rv[2]) * sc, __uint_as_float(rv[3]) * sc);
                    a.z = pack_bf16x2(__uint_as_float(rv[4]) * sc, __uint_as_float(rv[5]) * sc);
                    a.w = pack_bf16x2(__uint_as_float(rv[6]) * sc, __uint_as_float(rv[7]) * sc);
                    b.x = pack_bf16x2(__uint_as_float(rv[8]) * sc, __uint_as_float(rv[9]) * sc);
                    b.y = pack_bf16x2(__uint_as_float(rv[10]) * sc, __uint_as_float(rv[11]) * sc);
                    b.z = pack_bf16x2(__uint_as_float(rv[12]) * sc, __uint_as_float(rv[13]) * sc);
                    b.w = pack_bf16x2(__uint_as_float(rv[14]) * sc, __uint_as_float(rv[15]) * sc);
                    uint8_t* rowp = smem + C::offResW + (c >> 2) * (kTile * 128) + t * 128;
                    *reinterpret_cast<uint4*>(rowp + ((((2 * c) & 7) ^ (t & 7)) << 4)) = a;
                    *reinterpret_cast<uint4*>(rowp + ((((2 * c + 1) & 7) ^ (t & 7)) << 4)) = b;
                }
                fence_proxy_async_smem();
                rows_all(true);
                if (t == 0) {
#pragma unroll
                    for (int bb = 0; bb < C::kVB; ++bb)
                        tma_store_3d(&tm_out, smem + C::offResW + bb * (kTile * 128), bb * 64, r0, head);
                    tma_store_commit();
                    tma_store_wait<0>();
                }
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
    if (warp == 4) tmem_dealloc(tb, C::kCols);
    // one CTA holds the grid's end back until the grid before it is complete: what follows in the stream sees both
    if (MODE == kModeFwd && p.overlapped && blockIdx.x == gridDim.x - 1 && tid == 0)
        asm volatile("griddepcontrol.wait;" ::: "memory");
}

namespace {
// Block-wise path, between the passes.  state_scan_kernel: the per-block states of
// block_state_tc_kernel summed over the blocks before (suffix = 0) or after (suffix = 1) each
// block, as bf16 [BH x nblk][dvw][160] (tensor-core operand, transposed as the state kernel holds it) and fp32 row
// sums [BH x nblk][160].
__global__ void __launch_bounds__(256)
    state_scan_kernel(const float* __restrict__ part, const float* __restrict__ zpart, __nv_bfloat16* __restrict__ st,
                      float* __restrict__ sv, int nblk, int per, int suffix) {
    enter_dependent();
    const int e = blockIdx.x * 256 + threadIdx.x;
    const size_t h0 = (size_t)blockIdx.y * nblk;
    if (e < per) {
        float run = 0.f;
        for (int i = 0; i < nblk; ++i) {
            const int c = suffix ? nblk - 1 - i : i;
            st[(h0 + c) * per + e] = __float2bfloat16(run);
            run += part[(h0 + c) * per + e];
        }
    }
    if (blockIdx.x == 0 && threadIdx.x < 160) {
        float run = 0.f;
        for (int i = 0; i < nblk; ++i) {
            const int c = suffix ? nblk - 1 - i : i;
            sv[(h0 + c) * 160 + threadIdx.x] = run;
            run += zpart[(h0 + c) * 160 + threadIdx.x];
        }
    }
}
template <int DV, int KIND, int LT, bool XB = false>
based_status launch_pass(const CUtensorMap& n0, const CUtensorMap& w0, const CUtensorMap& n1, const CUtensorMap& w1,
                         const BParams& p, dim3 grid, const char* what, cudaStream_t stream,
                         const CUtensorMap* st = nullptr, const CUtensorMap* outm = nullptr) {
    constexpr int MODE = base_mode(KIND);
    using C = BCfg<DV, MODE, LT, XB>;
    static bool configured[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BASED_ERR_CUDA;
    {
        std::lock_guard<std::mutex> lock(setup_mutex());
        if (!configured[dev]) {
            if (cudaFuncSetAttribute(backward_tc_kernel<DV, KIND, LT, XB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)C::kSmem) != cudaSuccess)
                return BASED_ERR_CUDA;
            configured[dev] = true;
        }
    }
    // Dependent launches, but not the tile path's passes over the queries with more than a CTA per SM (d_v 112 / 128: per two SMs): theirs
    // would double up on the SMs that the grid ahead leaves first (us per backward call, no pass dependent / dk/dv / all: B2 H16 L1000
    // d_v128 43.9 / 43.0 / 44.8, B8 H12 L300 d_v64 18.7 / 18.8 / 19.3, B1 H8 L300 d_v128 18.8 / 17.8 / 17.0, B4 H16 L2048 d_v64, the keys' states
    // too, 97.6 / 95.9 / 95.1; dk/dv / all at d_v 128, 12 heads L1024 36.7 / 38.7, 16 37.2 / 39.6, 24 L768 30.9 / 32.3, 8 L1024 36.5 / 35.7, 16 L512
    // 22.4 / 21.6, at d_v 64 16 L1024 34.3 / 33.7)
    const bool dependent = MODE == kModeFwd ? p.overlapped || dependent_forward(grid.x, grid.x / p.heads, 4 * kSMs)
                                            : MODE == kModeDkDv || XB || grid.x <= (DV == 64 ? kSMs : kSMs / 2);
    const cudaError_t e = launch_ex(backward_tc_kernel<DV, KIND, LT, XB>, grid, dim3(kThreadsB), C::kSmem, 1, dependent, stream, n0, w0, n1,
                                    w1, st ? *st : n0, outm ? *outm : w0, p);
    note_launch();
    const based_status s2 = check_launch(what);
    return e == cudaSuccess ? s2 : BASED_ERR_CUDA;
}

// Block length of the block-wise path, or 0 for the tile path alone.  The block-wise path needs d' = 16 and the
// statistics in one sweep (the forward output, or the numerator-only form); its cost grows with L where the tile
// path's grows with L^2.  Tiles / blocks of 256 tokens on B200, us, around the lines below:
//   128 heads: d_v 64 L 768 63 / 70, L 1024 98 / 91; d_v 128 L 768 96 / 97, L 1024 142 / 129
//   64 heads: d_v 64 L 768 34 / 47, L 1024 52 / 54, L 1280 73 / 66; d_v 128 L 768 50 / 59, L 1024 74 / 72
//   16 heads: d_v 64 L 768 29 / 36, L 1024 36 / 37, L 1536 51 / 42; d_v 128 L 1280 46 / 52, L 1536 53 / 54, L 2048 70 / 55
//   32 heads: d_v 64 L 1280 46 / 61, L 1536 56 / 66, L 2048 82 / 70; d_v 128 L 1536 74 / 91, L 2048 112 / 101
// And, since both paths' passes are dependent launches, at d_v 64: 64 heads L 768 32 / 48, L 800 41 / 48 (blocks there all the same:
// the line of 64 heads and more is 128 heads'; up to some 110 heads and 1024 tokens tiles would be the faster), 80 L 768 43 / 49, 128 62 / 66, L 769 74.4 / 74.1, L 897 93 / 83; 8 heads L 769 28 / 34, L 1024 34 / 35, L 1025 36 / 35; 16 29 / 36, 34 / 35,
// 36 / 36; 24 30 / 36, 36 / 37, 38 / 37; 32 L 769 32 / 38, L 897 37.4 / 37.8, L 1024 39.2 / 37.9; 2 (where the line stays) L 768 26 / 28, L 769
// 28.0 / 28.8, L 897 31 / 29.  The tile path is also the more precise (2.3e-3 against 2.4e-3 of fp64 gradients), so no line moves below where it was.
// Below 64 heads one CTA per head and block sums the states, and a second short wave of those costs as much as a full one:
// there the line lies later once the blocks are more than one wave (24 heads are not at L 1536: 54 / 44, 60 / 56).
// With them at d_v 128 blocks of 512 tokens are the faster from 64 k rows on (256 / 512 tokens: 16 heads L 8192 217 / 206,
// L 16384 403 / 381, 32 heads L 4096 216 / 202; 8 heads L 4096 64 / 79, L 8192 117 / 116; 2 heads L 16384 73 / 83).  Blocks of
// 128 tokens are within 3 % at d_v 64 (64 heads L 2048 99 / 100, 200 heads 286 / 276) and lose at d_v 128 (128 heads 255 / 242).
// A caller without the forward output gets it recomputed into the workspace first (one forward pass, 20 us at B4 H16
// L2048 d_v64, 83 us at B8 H16 L4096 d_v128), from somewhat longer sequences on (d_v 64: 64 heads L 1024 62 / 67, L 1280
// 85 / 81, 128 heads L 1280 154 / 130; d_v 128: 64 heads L 1024 87 / 87, L 1280 122 / 107, 16 heads L 1536 70 / 71).
int backward_block_len(int L, int df, bool merged, int d_v, int BH) {
    if (df != 16) return 0;
    int from;
    if (BH >= 64) from = !merged ? 1280 : d_v == 64 ? 769 : 1024;
    else if (BH * ((L + 255) / 256) > kSMs) from = 2048;
    else from = d_v != 64 ? 1536 : !merged ? 1024 : BH <= 4 ? 768 : BH < 32 ? 1025 : 897;
    if (L < from) return 0;
    return BH < 64 && d_v != 64 && L >= 4096 && (long long)BH * L >= 65536 ? 512 : 256;
}
size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
struct BlockWs {
    float* sv; float* zpart; float* part; __nv_bfloat16* st;
    __nv_bfloat16* out; void* fwd;                   // the recomputed forward output and the forward pass's own scratch
    size_t bytes;
};
// scratch after the [BH, L] float2 statistics
BlockWs block_ws(float* ws, int BH, int L, int dvr, int nblk) {
    BlockWs w{};
    const uintptr_t base = reinterpret_cast<uintptr_t>(ws);
    size_t off = align256((size_t)BH * L * 8);
    w.sv = reinterpret_cast<float*>(base + off);     off = align256(off + (size_t)BH * nblk * 160 * 4);
    w.zpart = reinterpret_cast<float*>(base + off);  off = align256(off + (size_t)BH * nblk * 160 * 4);
    // the blocks' own fp32 sums: only where a scan adds them up (few heads)
    w.part = reinterpret_cast<float*>(base + off);   off = align256(off + (BH >= 64 ? 0 : (size_t)BH * nblk * 160 * dvr * 4));
    w.st = reinterpret_cast<__nv_bfloat16*>(base + off);  off = align256(off + (size_t)BH * nblk * 160 * dvr * 2);
    w.out = reinterpret_cast<__nv_bfloat16*>(base + off); off = align256(off + (size_t)BH * L * dvr * 2);
    w.fwd = reinterpret_cast<void*>(base + off);     off = align256(off + prefill_tc_workspace_bytes(BH, L, dvr));
    w.bytes = off;
    return w;
}

// Tile passes: whether the longest loops of all heads start first, for an even end and long loops beside short ones on an SM.
// Head by head the last heads' long loops start when the other SMs have run dry: the forward at B4 H16 L2048 d' 24 d_v 64 took
// 50 us against 39, at B4 H16 L16384 d_v 128, where the looped tiles of all heads are 300 MB and do not stay in L2, 3609
// against 3390; the backward at the first 230 against 187, at B2 H16 L1000 d_v 128 (256 CTAs) 63 against 49.  With a CTA or
// less per SM there is nothing to even out: head by head 18.5 against 19.4 (B1 H8 L300, d' 16).
int long_loops_first(int BH, int L) { return (long long)BH * ((L + kTile - 1) / kTile) > kSMs; }

template <int DV>
based_status launch_dvb(const void* q, const void* k, const void* v, const void* out, const void* g, int dout_H, void* dq, void* dk,
                        void* dv, float* ws, int BH, int L, int df, int dvr, int numerator_only, cudaStream_t stream) {
    constexpr int LTK = (DV == 64) ? 64 : 128;       // looped tile of the dk/dv pass (d_v 128 needs all 512 columns anyway)
    float2* stats = reinterpret_cast<float2*>(ws);
    // own tiles: 128 rows; looped tiles: 64 rows (and LTK rows for the dk/dv pass)
    CUtensorMap tq, tk, tv, tg, tk64, tv64, tqL, tgL, tdv;
    const CUtensorMapSwizzle s64 = CU_TENSOR_MAP_SWIZZLE_64B, s128 = CU_TENSOR_MAP_SWIZZLE_128B;
    auto dout_map = [&](CUtensorMap* m, int rows) { return make_head_rows_map_bf16(m, g, BH, dout_H, L, dvr, 64, rows, s128); };
    if (!make_rows_map_bf16(&tq, q, BH, L, df, 32, kTile, s64) || !make_rows_map_bf16(&tk, k, BH, L, df, 32, kTile, s64) ||
        !make_rows_map_bf16(&tv, v, BH, L, dvr, 64, kTile, s128) || !dout_map(&tg, kTile) ||
        !make_rows_map_bf16(&tk64, k, BH, L, df, 32, 64, s64) || !make_rows_map_bf16(&tv64, v, BH, L, dvr, 64, 64, s128) ||
        !make_rows_map_bf16(&tqL, q, BH, L, df, 32, LTK, s64) || !dout_map(&tgL, LTK) ||
        !make_rows_map_bf16(&tdv, dv, BH, L, dvr, 64, kTile, s128))
        return BASED_ERR_CUDA;
    BParams p{};
    if (error_word_ptr(&p.err) != BASED_OK) return BASED_ERR_CUDA;
    p.stats_in = stats;
    p.stats_out = stats;
    p.o_raw = static_cast<const __nv_bfloat16*>(out);
    p.dq = static_cast<__nv_bfloat16*>(dq);
    p.dk = static_cast<__nv_bfloat16*>(dk);
    p.L = L;
    p.dvw = dvr;
    p.numerator_only = numerator_only;
    p.df = df;
    p.kdim = df <= 16 ? 16 : 32;
    p.s1 = 1.0f / sqrtf((float)df);
    p.s2 = 0.5f / (float)df;
    const dim3 grid((unsigned)((L + kTile - 1) / kTile) * BH);
    p.heads = BH;
    p.by_length = long_loops_first(BH, L);
    p.dout_H = dout_H;
    based_status st;
    const int W = backward_block_len(L, df, out != nullptr || numerator_only, dvr, BH);
    if (W > 0) {
        // block-wise: pairs inside a block of W tokens by tiles, everything else through summed block states
        const int nblk = (L + W - 1) / W;
        const BlockWs w = block_ws(ws, BH, L, dvr, nblk);
        CUtensorMap tst;
        // the block states lie transposed, [BH x nblk][d_v][160]: boxes of 32 features x all value columns
        if (!make_rows_map_bf16(&tst, w.st, BH * nblk, dvr, 160, 32, 64 * BCfg<DV, kModeDkDv, LTK>::kVB, s64)) return BASED_ERR_CUDA;
        if (out == nullptr && !numerator_only) {
            // the centre of the merged pass: the forward output, recomputed
            st = launch_prefill_tc(q, k, v, w.out, nullptr, nullptr, BH, L, dvr, 0, w.fwd, stream);
            if (st != BASED_OK) return st;
            p.o_raw = w.out;
        }
        p.W = W;
        p.by_length = 0;                             // loops of one length
        p.nblk = nblk;
        p.sv = w.sv;
        // With many heads one CTA per head walks the blocks and writes the running sums; with few, one CTA per head
        // and block writes the block's own sums and a scan adds them up.
        const bool running = BH >= 64;
        auto states = [&](const void* x, const void* val, const void* sts, int rev) -> based_status {
            const int val_H = rev ? dout_H : 0;
            if (running) return launch_block_states_tc(x, val, sts, w.st, w.sv, nullptr, nullptr, BH, val_H, L, W, dvr, rev, stream);
            based_status s2 = launch_block_states_tc(x, val, sts, w.st, w.sv, w.part, w.zpart, BH, val_H, L, W, dvr, rev, stream);
            if (s2 != BASED_OK) return s2;
            // (dependent with many heads, and with one: with a few the pass behind it, a dependent launch itself, comes in while the scan's blocks
            // are being placed; us per backward call, dependent / plain: d_v 128 2 heads L3000 49.4 / 42.7, 6 L2048 49.3 / 42.6, 8 L1536 48.3 / 44.1,
            // 12 L2048 47.7 / 48.3, d_v 64 1 L1024 27.9 / 30.1, 4 L2048 35.4 / 32.1, 12 L1536 37.5 / 34.7, 16 L3000 61.5 / 62.2, 32 L2048 66.4 / 67.2)
            const bool dependent = BH == 1 || BH >= (DV == 64 ? 16 : 12);
            const cudaError_t e = launch_ex(state_scan_kernel, dim3((160 * dvr + 255) / 256, BH), dim3(256), 0, 1, dependent, stream, w.part,
                                            w.zpart, w.st, w.sv, nblk, 160 * dvr, rev);
            note_launch();
            s2 = check_launch("state_scan_kernel");
            return e == cudaSuccess ? s2 : BASED_ERR_CUDA;
        };
        // states of the keys: S = sum mono(k) v^T, z = sum mono(k), summed over the blocks before each block
        if ((st = states(k, v, nullptr, 0)) != BASED_OK) return st;
        st = launch_pass<DV, kModeDqS, 64, true>(tq, tg, tk64, tv64, p, grid, "backward_tc_kernel<stats+dq, blocks>", stream, &tst);
        if (st != BASED_OK) return st;
        // states of the queries: R = sum mono(q) (dout / D)^T, R_b = sum b mono(q), summed over the blocks after each block
        if ((st = states(q, g, stats, 1)) != BASED_OK) return st;
        if (DV == 128) {
            // 32-row looped tiles: the accumulators then fit 256 tensor-memory columns and two CTAs share an SM, which
            // hides the fixed latency of these short-lived CTAs (273 -> 220 us for the pass at B8 H16 L4096)
            CUtensorMap tq32, tg32;
            if (!make_rows_map_bf16(&tq32, q, BH, L, df, 32, 32, s64) || !dout_map(&tg32, 32)) return BASED_ERR_CUDA;
            return launch_pass<DV, kModeDkDv, 32, true>(tk, tv, tq32, tg32, p, grid, "backward_tc_kernel<dkdv, blocks>", stream, &tst,
                                                        &tdv);
        }
        return launch_pass<DV, kModeDkDv, LTK, true>(tk, tv, tqL, tgL, p, grid, "backward_tc_kernel<dkdv, blocks>", stream, &tst,
                                                     &tdv);
    }
    if (out != nullptr || numerator_only) {
        // statistics and dq in one sweep (needs the forward output as the centre of the packed products)
        st = launch_pass<DV, kModeDqS, 64>(tq, tg, tk64, tv64, p, grid, "backward_tc_kernel<stats+dq>", stream);
        if (st != BASED_OK) return st;
    } else {
        // statistics: own = queries (q, dout), looped = keys (k, v)
        st = launch_pass<DV, kModeStats, 64>(tq, tg, tk64, tv64, p, grid, "backward_tc_kernel<stats>", stream);
        if (st != BASED_OK) return st;
        // dq: own = queries (q, dout), looped = keys (k, v)
        st = launch_pass<DV, kModeDq, 64>(tq, tg, tk64, tv64, p, grid, "backward_tc_kernel<dq>", stream);
        if (st != BASED_OK) return st;
    }
    // dk, dv: own = keys (k, v), looped = queries (q, dout)
    return launch_pass<DV, kModeDkDv, LTK>(tk, tv, tqL, tgL, p, grid, "backward_tc_kernel<dkdv>", stream, nullptr, &tdv);
}
}  // namespace

// Forward of the definition form, for feature dimensions other than 16 and one chunk of d' 16 (bf16 io,
// empty initial state); on the same tiles: out = (sum_j w_ij v_j) / (sum_j w_ij + eps), w = 1 + s/sqrt(d') + s^2/(2 d').
// The weights lie over the scores, so at d_v 64 a CTA takes 128 columns of tensor memory and four share an SM, and tiles off
// the diagonal evaluate two pairs per instruction: B4 H16 L2048 d_v64 80 -> 48 us (looped tiles of 128 rows: 47), 38 with the
// longest loops first (36.7 with the scores' second half loaded ahead).  With the state asked for it is launched beside that
// kernel, which takes 16 us alone; the call 55 (one after the other, and both kernels slower, 80 + 61 before).
based_status launch_quadratic_forward_tc(const void* q, const void* k, const void* v, void* out, int BH, int L,
                                         int d_feat, int d_v, int numerator_only, bool overlapped, cudaStream_t stream) {
    // Two groups of row warps on one tile after the other (quadratic_fwd_tc.cu) where that is the faster: at d_v 128 always, at d_v 64
    // where its two CTAs per SM hold every tile, or few heads' long loops leave this kernel's four unfilled (us at d' 24, this / that:
    // d_v 128 L16 with 1 head 4.5 / 3.6, with 1024 15.4 / 14.3, L64 16.5 / 15.7; d_v 64 with 64 heads L64 3.5 / 3.5, L128 4.3 / 3.9, with
    // 148 4.9 / 4.2, with 400 7.1 / 8.5, L300 17.0 / 21.7, with 32 L1536 19.4 / 13.9, with 20 L2048 22.2 / 16.6, with 64 L1024 18.0 / 14.3,
    // L1536 22.5 / 23.6, L4096 113 / 111).  One rule with the state beside it and without, so that the outputs are the same bits (with
    // it, 64 heads L64 6.9 / 7.4, L128 8.2 / 7.9, L1024 20.4 / 21.4, 32 heads L1536 22.4 / 19.4).
    const long long tiles = (long long)((L + kTile - 1) / kTile) * BH;
    if (d_v != 64 || (L > 64 && tiles <= 2 * kSMs) || (L > 11 * kTile && tiles <= 4 * kSMs))
        return launch_quadratic_groups_tc(q, k, v, out, BH, L, d_feat, d_v, numerator_only, overlapped, stream);
    CUtensorMap tq, tk64, tv64, tout;
    const CUtensorMapSwizzle s64 = CU_TENSOR_MAP_SWIZZLE_64B, s128 = CU_TENSOR_MAP_SWIZZLE_128B;
    if (!make_rows_map_bf16(&tq, q, BH, L, d_feat, 32, kTile, s64) || !make_rows_map_bf16(&tk64, k, BH, L, d_feat, 32, 64, s64) ||
        !make_rows_map_bf16(&tv64, v, BH, L, d_v, 64, 64, s128) || !make_rows_map_bf16(&tout, out, BH, L, d_v, 64, kTile, s128))
        return BASED_ERR_CUDA;
    BParams p{};
    if (error_word_ptr(&p.err) != BASED_OK) return BASED_ERR_CUDA;
    p.L = L;
    p.dvw = d_v;
    p.overlapped = overlapped;
    p.numerator_only = numerator_only;
    p.df = d_feat;
    p.kdim = d_feat <= 16 ? 16 : 32;
    p.s1 = 1.0f / sqrtf((float)d_feat);
    p.s2 = 0.5f / (float)d_feat;
    const dim3 grid((unsigned)((L + kTile - 1) / kTile) * BH);
    p.heads = BH;
    p.by_length = long_loops_first(BH, L);
    if (d_feat == 16) return launch_pass<64, kModeFwdRounded, 64>(tq, tq, tk64, tv64, p, grid, "quadratic forward (tc)", stream, nullptr, &tout);
    return launch_pass<64, kModeFwd, 64>(tq, tq, tk64, tv64, p, grid, "quadratic forward (tc)", stream, nullptr, &tout);
}

int backward_tc_block_tokens(int BH, int L, int d_feat, int d_v, int merged) {
    return backward_block_len(L, d_feat, merged != 0, d_v, BH);
}

size_t backward_tc_workspace_bytes(int BH, int L, int d_v) {
    // with the forward output or without: neither line lies below the other everywhere (5 to 31 heads, d_v 64: 1025 with, 1024 without)
    const int with = backward_block_len(L, 16, true, d_v, BH), W = with ? with : backward_block_len(L, 16, false, d_v, BH);
    if (W > 0) return block_ws(nullptr, BH, L, d_v, (L + W - 1) / W).bytes;         // statistics, block states
    return (size_t)BH * L * 2 * sizeof(float);                 // (1 / D, b) per row
}

based_status launch_prefill_backward_tc(const void* q, const void* k, const void* v, const void* out, const void* g, int dout_H,
                                        void* dq, void* dk, void* dv, float* ws, int BH, int L, int d_feat, int d_v,
                                        int numerator_only, cudaStream_t stream) {
    if (d_v == 64) return launch_dvb<64>(q, k, v, out, g, dout_H, dq, dk, dv, ws, BH, L, d_feat, 64, numerator_only, stream);
    return launch_dvb<128>(q, k, v, out, g, dout_H, dq, dk, dv, ws, BH, L, d_feat, d_v, numerator_only, stream);  // 112 or 128
}

}  // namespace based

#ifdef BASED_TRACE
// debug builds: which barrier each warp of the first CTA that gave up was waiting on (this file's copy)
extern "C" void based_debug_read_waits_bwd(unsigned int* out) {
    cudaDeviceSynchronize();
    cudaMemcpyFromSymbol(out, based::sm100::g_wait_dbg, sizeof(unsigned int) * 128);
    cudaMemcpyFromSymbol(out + 128, based::sm100::g_wait_owner, sizeof(unsigned int));
    unsigned int zero[129] = {};
    cudaMemcpyToSymbol(based::sm100::g_wait_dbg, zero, sizeof(unsigned int) * 128);
    cudaMemcpyToSymbol(based::sm100::g_wait_owner, zero, sizeof(unsigned int));
}
#endif
