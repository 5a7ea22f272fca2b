// Definition form of the causal Taylor linear attention (left-hand side of Eq. (2) of Sec. 4.1, d' = 16) for fp32 io on the
// tensor cores: the forward pass from the empty state, and the backward pass at d_v 64.
//
// Every fp32 operand x is three bf16 parts, x = x0 + x1 + x2 (each the rounding of what the parts before it leave: 24 bits
// in all), and a product of two operands the six products of parts (a, b) with a + b <= 2; what is left out is below 2^-25
// of it.  The products of parts are exact and tcgen05.mma adds them up in fp32, but it cuts what it adds off at the
// accumulator's last place instead of rounding it, so a sum that is carried through many instructions drifts towards zero
// (one accumulator for K = 1024: 7e-6 in the 2-norm, fp32 multiply-adds 6e-7).  Hence
//   - within a tile the small products go first: only the last four instructions meet an accumulator of full size;
//   - no accumulator of the products of first parts lives longer than one looped tile of 64 rows: it is added to fp32
//     registers, rounding (K = 64: 7e-8 against 1.5e-7 of fp32 multiply-adds, K = 1024: 1.0e-7 against 5.7e-7).
// The parts are those of 2^24 x: of x below 2^-109 the third part, and further down the second, would have bits below the last
// bf16 subnormal (v or dout of 1e-36: 2.7e-5 off).  Scores and products of dout and v carry 2^48: the polynomials' coefficients
// take that back.  What is split again (weights times dout . v, times 1/D) is formed at 2^24 of its size, for the same
// reason, and the results are scaled back at the end.  All of it by powers of two: nothing is rounded.
//
// One CTA per (head, 128 own rows), looping over tiles of 64 rows of the other side; formulas as in backward_f32.cu:
//   kFwd   own = queries, looped = keys:   Y += W V,  W = 1 + S/4 + S^2/32, S = Q K^T
//   kDq    own = queries, looped = keys:   X += W' (G V^T - m) K,  Y += W' K,  row sums of W and W (G V^T)
//   kKeys  own = keys, looped = queries:   dK += DS^T Q,  dV += W^T (G / D)
// The parts are written by a kernel ahead (split_parts_kernel) and come by TMA.  Split inside the loop, every looped tile once
// per own tile, they took 40 % of the instructions.
// In a backward tile the scores alone give half of the weights: their products start while the rows form the other half.
// Three warpgroups and some warps.  Two groups of rows (a TMEM lane per thread): weights, masks, row sums, and the parts of
// the weights back to tensor memory as A operands; forward: the groups take the looped tiles in turn, backward: half of each
// tile's columns each.  One group collects: it adds every tile's accumulator to its registers and writes the results.  One
// warp issues the scores' MMAs, one the products', converged with one elected lane (a warp that has issued a tile's MMAs goes
// on only when the last of them has left the queue, so one for both let the tensor pipe run dry twice per tile: forward at B1 H2
// L4096 55.6 -> 52.0 us); one the loads.
//
// Infinities, NaN and values from 2^104 on do not split (inf - inf is NaN), scores or products of dout and v from 2^80 on overflow
// at 2^48 of their size, and a masked weight of zero times infinity is NaN in rows that do not see the key.  Either way what
// comes out is not finite: such rows are computed once more with plain fp32 multiply-adds, masked pairs left out (B2 H16 L1024 with a value of NaN in each head: 330 and 1000 us).
//
// Measured at B2 H16 L1024 d_v 64, against fp32 multiply-adds: forward 72 -> 28 us, backward 269 -> 80, errors in the 2-norm 0.8e-7
// for 1.9e-7 (outputs), 1.7e-7 for 2.8e-7 (dq), 1.9e-7 for 4.1e-7 (dk), 1.4e-7 for 7.6e-7 (dv).  The SMs are active for 39 k, 60 k and
// 68 k cycles of 15.6 looped tiles each, the tensor pipe in 38, 35 and 44 % of them.  What bounds them: an MMA with both operands in shared memory is read at 128 bytes per cycle, 48
// cycles at N = 64 where the tensor pipe needs 32, so the 30 of a tile's scores and products take 1440 cycles, those of dk and dv
// 990.  The 256 CTAs of such a call are 1.7 waves, with some 8 k cycles of start and end each.  480 threads leave 128 registers:
// the forward for d_v 112 and 128, whose collectors hold 128 sums a thread, spills 0.9 KB, dq 0.1 KB.
#include <cooperative_groups.h>

#include <mutex>
#include <type_traits>
#include <utility>

#include "common.cuh"
#include "sm100.cuh"

namespace based {
using namespace sm100;

namespace {
namespace cg = cooperative_groups;

constexpr int kOwn = 128, kLT = 64;
constexpr int kNThreads = 480;
constexpr int kFwd = 0, kDq = 1, kKeys = 2;
constexpr float kUp = 0x1p24f, kDown = 0x1p-24f, kDown2 = 0x1p-48f;    // of the parts' scale; of the scale of a product of two
// parts (a, b) of the six products, the smallest first
__host__ __device__ constexpr int part_a(int i) { return i < 3 ? i : i == 4; }
__host__ __device__ constexpr int part_b(int i) { return i < 3 ? 2 - i : i == 3; }

template <int DV, int MODE> struct QCfg {
    static constexpr bool kBwd = MODE != kFwd;
    static constexpr int kVB = DV / 64;                                // 64-column blocks of a wide tile
    // shared memory: tiles of 128-byte rows, SWIZZLE_128B.  Narrow (q, k): the parts' 16 columns side by side, 48 of 64
    // columns used.  Wide (v, dout): a tile per part, [kVB][rows][64].
    static constexpr uint32_t kOwnPart = kVB * kOwn * 128, kPart = kVB * kLT * 128, kNarrow = kLT * 128;
    static constexpr uint32_t offOwnN = 0, offOwnW = kOwn * 128, offStage = offOwnW + (kBwd ? 3 * kOwnPart : 0);
    static constexpr uint32_t kStage = kNarrow + 3 * kPart;
    static constexpr int kNS = kBwd ? 4 : DV == 64 ? 6 : 3;
    static constexpr uint32_t offStats = offStage + kNS * kStage;      // keys pass: inv, then b (QParams), of a stage's queries
    static constexpr uint32_t offSum = offStats + (MODE == kKeys ? kNS * kLT * 8 : 0);                // row sums of the two row groups
    static constexpr uint32_t offBars = offSum + 2 * kOwn * 8;
    static constexpr uint32_t kSmem = offBars + 512 + 1024;
    // tensor memory: sets of (scores, dout.v products, room): the weights' parts take their place, 32 columns a tensor; the
    // accumulators
    static constexpr uint32_t kSet = kBwd ? 192 : 96;
    static constexpr int kNSet = !kBwd && DV == 64 ? 4 : 2;
    static constexpr int kNAcc = MODE == kKeys ? 1 : 2;
    // Y, two in turn; dV; of X, Y, dK the products of first parts in 16 columns (X, Y: two in turn), those of the others in
    // two times 16 (colRest)
    static constexpr uint32_t colAcc = kNSet * kSet, colAcc2 = colAcc + 64;
    static constexpr uint32_t kAcc = MODE == kDq ? 16 : DV;            // from one of two in turn to the other
    static constexpr uint32_t colRest = colAcc + 32, colRest2 = colAcc2 + (MODE == kDq ? 32 : 16);
    static_assert(kBwd ? DV == 64 && colRest2 + 32 <= 512 : colAcc + 2 * DV <= 512, "tensor memory budget");
    // column of K-step k (16 looped rows) of part u of the weights in a set.  The first weights (t = 0: W, kDq: W') need the
    // scores alone and lie over them, the second (kDq: W' (GV - m), kKeys: DS) over the products; third parts in the room behind
    static __host__ __device__ constexpr uint32_t weight_col(int t, int u, int k) {
        return kBwd ? (u < 2 ? 64 * t + 16 * k + 8 * u : 128 + 16 * k + 8 * t) : u < 2 ? 16 * k + 8 * u : 64 + 8 * k;
    }
};

enum { bOwn = 0, bFull = 1, bEmpty = 7, bScore = 13, bWeight = 17, bSetFree = 21, bAccDone = 25, bAccFree = 27, bScoreG = 29, bWeightB = 31, bCount = 33 };

struct QParams {
    const float *own_n, *own_w, *loop_n, *loop_w;    // narrow and wide tensors of the own and the looped side (forward: own_w unused)
    float *inv, *b;                                  // kUp / D and -(G V^T's mean under the weights) per query, [heads][pitch]:
                                                     // written by kDq, read by kKeys
    const float* m;                                  // kDq: the centres m_i = G_i.v_i, [heads][L]
    int pitch;                                       // L rounded up to whole looped tiles
    float *out_n, *out_w;                            // dq or dk; the forward output or dv
    // dout may lie [B, L, H, d_v] (own side of kDq, looped side of kKeys): then H, and the slab's first head; else H = 0
    int dout_H, dout_h0;
    unsigned int* err;
    int heads, L, dvw, numerator_only, by_length, nsplit;   // nsplit: CTAs of a cluster that share an own tile's loop
};

__device__ __forceinline__ uint64_t f2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t bits2(uint32_t a, uint32_t b) { return f2(__uint_as_float(a), __uint_as_float(b)); }
// the three bf16 parts of a pair
__device__ __forceinline__ void split_pair(uint64_t x, uint32_t& p0, uint32_t& p1, uint32_t& p2) {
    const uint64_t minus = f2(-1.f, -1.f);
    auto round = [](uint64_t v) {
        float lo, hi;
        unpack2(v, lo, hi);
        const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<const uint32_t*>(&h);
    };
    auto wide = [](uint32_t p) { return f2(__uint_as_float(p << 16), __uint_as_float(p & 0xffff0000u)); };
    p0 = round(x);
    x = fma2(wide(p0), minus, x);
    p1 = round(x);
    x = fma2(wide(p1), minus, x);
    p2 = round(x);
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// AND over rows and collectors; orders their shared-memory accesses
__device__ __forceinline__ bool workers_all(bool pred) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, 384, p;\n\t"
        "selp.b32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)pred)
        : "memory");
    return r != 0;
}
// a whole 32-byte sector per lane; arrays that lie on 16 bytes only: two halves
__device__ __forceinline__ void store8(float* dst, const float (&x)[8]) {
    if (reinterpret_cast<uintptr_t>(dst) & 31) {
        reinterpret_cast<float4*>(dst)[0] = make_float4(x[0], x[1], x[2], x[3]);
        reinterpret_cast<float4*>(dst)[1] = make_float4(x[4], x[5], x[6], x[7]);
        return;
    }
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]),
                 "f"(x[4]), "f"(x[5]), "f"(x[6]), "f"(x[7])
                 : "memory");
}

// offset of a head's first row of dout and the distance of its rows
__device__ __forceinline__ size_t dout_rows(int H, int h0, size_t head, int L, int W, int& pitch) {
    pitch = W;
    if (H == 0) return head * (size_t)L * W;
    pitch = H * W;
    const size_t g = h0 + head, b = g / H;
    return (b * L * H + (g - b * H)) * W;
}
// The rows of a warp, a lane each, by plain multiply-adds, pair by pair: the narrow results (dq, dk) of lanes with need_n, the
// wide ones (the output, dv) of those with need_w.  buf: kPlainFloats of shared memory of the warp's own, for 32 looped rows at a
// time.
constexpr int kPlainPitch = kDFeat + 64 + 4;         // narrow row, wide columns, 1/D, minus the mean
constexpr int kPlainFloats = 32 * kPlainPitch;
template <int MODE>
__device__ __noinline__ void plain_rows(const QParams& p, float* buf, size_t head, int row, bool need_n, bool need_w) {
    const int r = min(row, p.L - 1), W = p.dvw, L = p.L, lane = threadIdx.x & 31;
    const size_t hn = head * (size_t)L * kDFeat, hw = head * (size_t)L * W, hs = head * (size_t)p.pitch;
    const int from = MODE == kKeys ? __reduce_min_sync(~0u, r) : 0, to = MODE == kKeys ? L - 1 : __reduce_max_sync(~0u, r);
    int own_pitch = W, loop_pitch = W;
    const float* own_w = MODE == kFwd ? nullptr : p.own_w + (MODE == kDq ? dout_rows(p.dout_H, p.dout_h0, head, L, W, own_pitch) : hw);
    const float *loop_n = p.loop_n + hn,
                *loop_w = p.loop_w + (MODE == kKeys ? dout_rows(p.dout_H, p.dout_h0, head, L, W, loop_pitch) : hw);
    float xn[kDFeat];
    auto row4 = [](float (&d)[kDFeat], const float* src) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float4 u = *reinterpret_cast<const float4*>(src + 4 * e);
            d[4 * e] = u.x; d[4 * e + 1] = u.y; d[4 * e + 2] = u.z; d[4 * e + 3] = u.w;
        }
    };
    row4(xn, p.own_n + hn + (size_t)r * kDFeat);
    auto dot16 = [](const float (&a)[kDFeat], const float (&b)[kDFeat]) {
        float s = 0.f, t = 0.f;
#pragma unroll
        for (int e = 0; e < kDFeat; e += 2) {
            s = fmaf(a[e], b[e], s);
            t = fmaf(a[e + 1], b[e + 1], t);
        }
        return s + t;
    };
    auto weight = [](float s) { return fmaf(s, fmaf(s, 0.03125f, 0.25f), 1.0f); };
    // 32 looped rows from j on, `cols` wide columns from c on
    auto stage = [&](int j, int c, int cols) {
        __syncwarp();
        for (int e = lane; e < 32 * 4; e += 32) {
            const int t = min(j + (e >> 2), L - 1), u = 4 * (e & 3);
            *reinterpret_cast<float4*>(buf + (e >> 2) * kPlainPitch + u) = __ldg(reinterpret_cast<const float4*>(loop_n + (size_t)t * kDFeat + u));
        }
        for (int e = lane; e < 8 * cols; e += 32) {
            const int i = e / (cols / 4), t = min(j + i, L - 1), u = 4 * (e % (cols / 4));
            *reinterpret_cast<float4*>(buf + i * kPlainPitch + kDFeat + u) = __ldg(reinterpret_cast<const float4*>(loop_w + (size_t)t * loop_pitch + c + u));
        }
        if (MODE == kKeys) {
            const int t = min(j + lane, L - 1);
            buf[lane * kPlainPitch + kDFeat + 64] = p.inv[hs + t] * kDown;
            buf[lane * kPlainPitch + kDFeat + 65] = p.b[hs + t];
        }
        __syncwarp();
    };
    float den = 0.f;
    if (MODE != kFwd && __any_sync(~0u, need_n)) {
        constexpr int DV = 64;
        const float* own = own_w + (size_t)r * own_pitch;
        float m = 0.f, num = 0.f, x[kDFeat] = {}, y[kDFeat] = {};
        if (MODE == kDq && !p.numerator_only)
            for (int c = 0; c < DV; ++c) m = fmaf(own[c], loop_w[(size_t)r * DV + c], m);
        float g[DV / kDFeat][kDFeat];
#pragma unroll
        for (int c = 0; c < DV / kDFeat; ++c) row4(g[c], own + c * kDFeat);
        for (int j0 = from; j0 <= to; j0 += 32) {
            stage(j0, 0, DV);
            for (int i = 0; i < 32 && j0 + i <= to; ++i) {
                const float* at = buf + i * kPlainPitch;
                float nj[kDFeat], d[kDFeat], gv = 0.f;
                row4(nj, at);
#pragma unroll
                for (int c = 0; c < DV / kDFeat; ++c) {
                    row4(d, at + (c + 1) * kDFeat);
                    gv += dot16(g[c], d);
                }
                const float s = dot16(xn, nj), w1 = fmaf(s, 0.0625f, 0.25f);
                if (MODE == kKeys ? j0 + i < r : j0 + i > r) continue;
                const float a = MODE == kDq ? w1 * (gv - m) : (gv + at[kDFeat + 65]) * at[kDFeat + 64] * w1;
                if (MODE == kDq) {
                    den += weight(s);
                    num = fmaf(weight(s), gv, num);
                }
#pragma unroll
                for (int e = 0; e < kDFeat; ++e) {
                    x[e] = fmaf(a, nj[e], x[e]);
                    if (MODE == kDq) y[e] = fmaf(w1, nj[e], y[e]);
                }
            }
        }
        const float inv = p.numerator_only ? 1.f : 1.f / (den + kEps), mean = p.numerator_only ? 0.f : num * inv;
        const float c = p.numerator_only ? 0.f : fmaf(m, inv, -mean * inv);
        if (need_n) {
#pragma unroll
            for (int e = 0; e < kDFeat; ++e) p.out_n[hn + (size_t)r * kDFeat + e] = MODE == kDq ? fmaf(x[e], inv, c * y[e]) : x[e];
            if (MODE == kDq) {
                p.inv[hs + r] = inv * kUp;
                p.b[hs + r] = -mean;
            }
        }
    }
    // 32 columns at a time; 112: the last 16 twice
    for (int c0 = 0; c0 < (MODE != kDq && __any_sync(~0u, need_w) ? W : 0); c0 += 32) {
        const int c = min(c0, W - 32);
        float y[2][kDFeat] = {};
        den = 0.f;
        for (int j0 = from; j0 <= to; j0 += 32) {
            stage(j0, c, 32);
#pragma unroll 2
            for (int i = 0; i < 32; ++i) {
                const float* at = buf + i * kPlainPitch;
                float nj[kDFeat], d[2][kDFeat];
                row4(nj, at);
#pragma unroll
                for (int h = 0; h < 2; ++h) row4(d[h], at + (h + 1) * kDFeat);
                float w = weight(dot16(xn, nj));
                if (MODE == kKeys) w *= at[kDFeat + 64];
                if (j0 + i > to || (MODE == kKeys ? j0 + i < r : j0 + i > r)) continue;
                den += w;
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int e = 0; e < kDFeat; ++e) y[h][e] = fmaf(w, d[h][e], y[h][e]);
            }
        }
        if (need_w)
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int e = 0; e < kDFeat; ++e)
                    p.out_w[hw + (size_t)r * W + c + h * kDFeat + e] = MODE == kKeys || p.numerator_only ? y[h][e] : y[h][e] / (den + kEps);
    }
}

// fp32 rows of W values as bf16 rows of 3 W: the first parts, the second, the third.  dout is read as it comes back from a
// projection, the heads of a token side by side: no copy ahead (5 us of a training step at B2 H16 L1024).  A block takes 1024 pieces of eight
// values of one tensor, four per thread, all loads under way at once.
struct SplitSet {
    const float* src[4];
    __nv_bfloat16* dst[4];
    unsigned pieces[4];                              // W / 8
    unsigned end[4];                                 // blocks of the tensors up to and with this one
    long long total[4];                              // pieces of the tensor
    float* m;                                        // products of the third and the fourth tensor's rows (d_v 64)
    unsigned L, H, h0;                               // the fourth tensor lies [B, L, H, W], h0 the slab's first head; H = 0: as the others
};
constexpr int kSplitPer = 4, kSplitBlock = 256 * kSplitPer;
__global__ void __launch_bounds__(256) split_parts_kernel(const SplitSet s) {
    asm volatile("griddepcontrol.wait;" ::: "memory");                 // the scratch may be in use up to there
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int i = 0;
    while (blockIdx.x >= s.end[i]) ++i;
    const unsigned block = blockIdx.x - (i > 0 ? s.end[i - 1] : 0), n = s.pieces[i];
    const long long e0 = (long long)block * kSplitBlock, left = s.total[i] - e0;
    const long long row0 = e0 / n;
    const unsigned c0 = (unsigned)(e0 - row0 * n);
    const float4* src = reinterpret_cast<const float4*>(s.src[i]);
    const bool strided = i == 3 && s.H != 0;
    auto at = [&](unsigned e) -> long long {         // piece e of the block
        if (!strided) return e0 + e;
        const unsigned row = (unsigned)row0 + (c0 + e) / n, c = (c0 + e) % n, g = row / s.L, l = row - g * s.L;
        const unsigned b = (s.h0 + g) / s.H, h = s.h0 + g - b * s.H;
        return (((long long)b * s.L + l) * s.H + h) * n + c;
    };
    uint4* dst = reinterpret_cast<uint4*>(s.dst[i]) + row0 * (3 * n);
    float4 a[kSplitPer], b[kSplitPer];
#pragma unroll
    for (int u = 0; u < kSplitPer; ++u) {
        const unsigned e = u * 256 + threadIdx.x;
        if (e < left) {
            const long long from = 2 * at(e);
            a[u] = __ldg(src + from);
            b[u] = __ldg(src + from + 1);
        }
    }
#pragma unroll
    for (int u = 0; u < kSplitPer; ++u) {
        const unsigned e = u * 256 + threadIdx.x;
        if (e >= left) break;
        const unsigned row = (c0 + e) / n, c = c0 + e - row * n;
        const uint64_t x[4] = {f2(a[u].x, a[u].y), f2(a[u].z, a[u].w), f2(b[u].x, b[u].y), f2(b[u].z, b[u].w)}, up = f2(kUp, kUp);
        uint32_t o[3][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) split_pair(mul2(x[k], up), o[0][k], o[1][k], o[2][k]);
#pragma unroll
        for (int k = 0; k < 3; ++k) dst[row * (3 * n) + c + k * n] = make_uint4(o[k][0], o[k][1], o[k][2], o[k][3]);
        if (i == 3 && s.m) {                         // eight lanes per row, rows in whole (d_v 64: eight pieces)
            const float4* w = reinterpret_cast<const float4*>(s.src[2]) + 2 * (e0 + e);
            const float4 g = a[u], h = b[u], v0 = __ldg(w), v1 = __ldg(w + 1);
            float m = fmaf(g.x, v0.x, fmaf(g.y, v0.y, fmaf(g.z, v0.z, g.w * v0.w)));
            m += fmaf(h.x, v1.x, fmaf(h.y, v1.y, fmaf(h.z, v1.z, h.w * v1.w)));
            const unsigned lanes = 0xffu << (threadIdx.x & 24);
#pragma unroll
            for (int k = 1; k < 8; k <<= 1) m += __shfl_xor_sync(lanes, m, k);
            if (c == 0) s.m[row0 + row] = m;
        }
    }
}
}  // namespace

template <int DV, int MODE>
__global__ void __launch_bounds__(kNThreads, 1)
    quadratic_f32_tc_kernel(const __grid_constant__ CUtensorMap tm_own_n, const __grid_constant__ CUtensorMap tm_own_w,
                            const __grid_constant__ CUtensorMap tm_loop_n, const __grid_constant__ CUtensorMap tm_loop_w,
                            const QParams p) {
    using C = QCfg<DV, MODE>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::offBars);
    uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(bars + bCount);
    volatile uint32_t* abort_flag = tmem_base_s + 1;
    float2* s_sum = reinterpret_cast<float2*>(smem + C::offSum);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ntiles = (p.L + kOwn - 1) / kOwn;
    // own tile: the longest loops first
    const int cta = blockIdx.x / p.nsplit, rank = blockIdx.x - cta * p.nsplit;
    const int turn = p.by_length ? cta / p.heads : cta % ntiles;
    const size_t head = p.by_length ? cta - turn * p.heads : cta / ntiles;
    const int own = MODE == kKeys ? turn : ntiles - 1 - turn;
    const int r0 = own * kOwn;
    const int begin = MODE == kKeys ? r0 / kLT : 0;
    const int count = (MODE == kKeys ? p.L - 1 : min(p.L, r0 + kOwn) - 1) / kLT - begin + 1;
    const int first = begin + count * rank / p.nsplit, n = begin + count * (rank + 1) / p.nsplit - first;      // (n = 0 is possible)
    const size_t hn = head * (size_t)p.L * kDFeat, hw = head * (size_t)p.L * p.dvw, hs = head * (size_t)p.pitch;

    if (tid == 0) {
        mbar_init(&bars[bOwn], 1);
#pragma unroll
        for (int i = 0; i < 6; ++i) {
            mbar_init(&bars[bFull + i], 1);
            mbar_init(&bars[bEmpty + i], 1);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            mbar_init(&bars[bScore + i], 1);
            mbar_init(&bars[bSetFree + i], 1);
            mbar_init(&bars[bWeight + i], C::kBwd ? 256 : 128);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            mbar_init(&bars[bAccDone + i], 1);
            mbar_init(&bars[bAccFree + i], 128);
            mbar_init(&bars[bScoreG + i], 1);
            mbar_init(&bars[bWeightB + i], 256);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 12) {
        tmem_alloc(tmem_base_s, 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = *tmem_base_s;
    bool ok = true;
    asm volatile("griddepcontrol.wait;" ::: "memory");                 // the parts; kKeys: inv and b
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    if (warp == 12 || warp == 14) {
        // ============================================================================ MMA warps: scores, products
        constexpr uint64_t dK = make_smem_desc_base(16, 1024, kSwizzle128B);                // K-major, or MN-major one block
        constexpr uint64_t dM = make_smem_desc_base(kLT * 128, 1024, kSwizzle128B);         // looped wide tile, MN-major
        constexpr uint32_t iS = make_idesc_bf16(128, kLT, 0, 0);
        constexpr uint32_t iW = make_idesc_bf16(128, DV, 0, 1);
        constexpr uint32_t i16 = make_idesc_bf16(128, 16, 0, 1), i32 = make_idesc_bf16(128, 32, 0, 1);
        const uint32_t lead = elect_one();
        // (in a cluster the address carries the CTA's rank above the descriptor's field)
        const uint32_t at0 = (smem_u32(smem) >> 4) & 0x3fffu, aOwnN = at0 + (C::offOwnN >> 4), aOwnW = at0 + (C::offOwnW >> 4);
        auto stage_at = [&](int t) { return at0 + ((C::offStage + (t % C::kNS) * C::kStage) >> 4); };
        auto scores = [&](int t) -> bool {
            if (!mbar_wait(&bars[bFull + t % C::kNS], (t / C::kNS) & 1, abort_flag) ||
                (t >= C::kNSet && !mbar_wait(&bars[bSetFree + t % C::kNSet], (t / C::kNSet - 1) & 1, abort_flag)))
                return false;
            tc_fence_after();
            const uint32_t aN = stage_at(t), aW = aN + (C::kNarrow >> 4), set = tb + (t % C::kNSet) * C::kSet;
#pragma unroll
            for (int i = 0; i < 6; ++i) {
                const uint32_t oa = desc_lo(dK) + aOwnN + 2 * part_a(i), ob = desc_lo(dK) + aN + 2 * part_b(i);
                if (i == 0) mma_ss_w<false>(lead, set, oa, desc_hi(dK), ob, desc_hi(dK), iS);
                else mma_ss_w<true>(lead, set, oa, desc_hi(dK), ob, desc_hi(dK), iS);
            }
            mma_commit_w(lead, &bars[bScore + t % C::kNSet]);
            if (C::kBwd) {
#pragma unroll
                for (int i = 0; i < 6; ++i)
#pragma unroll
                    for (int kk = 0; kk < DV / 16; ++kk) {
                        const uint32_t oa = desc_lo(dK) + aOwnW + ((part_a(i) * C::kOwnPart) >> 4) + 2 * kk;
                        const uint32_t ob = desc_lo(dK) + aW + ((part_b(i) * C::kPart) >> 4) + 2 * kk;
                        if (i == 0 && kk == 0) mma_ss_w<false>(lead, set + kLT, oa, desc_hi(dK), ob, desc_hi(dK), iS);
                        else mma_ss_w<true>(lead, set + kLT, oa, desc_hi(dK), ob, desc_hi(dK), iS);
                    }
                mma_commit_w(lead, &bars[bScoreG + t % C::kNSet]);
            }
            return true;
        };
        // acc += weights T x a looped narrow tile: products of first parts to 16 columns that start anew with every tile, the
        // others to two times 16 columns (by size) that live through the loop
        auto narrow = [&](auto weights_tag, uint32_t set, uint32_t acc, uint32_t rest, uint32_t aN, bool start) {
            constexpr int T = decltype(weights_tag)::value;
#pragma unroll
            for (int k = 0; k < kLT / 16; ++k) {
                const uint32_t b = desc_lo(dK) + aN + 128 * k;
                if (k == 0) mma_ts_w<false>(lead, acc, set + C::weight_col(T, 0, k), b, desc_hi(dK), i16);
                else mma_ts_w<true>(lead, acc, set + C::weight_col(T, 0, k), b, desc_hi(dK), i16);
                if (k == 0 && start) mma_ts_w<false>(lead, rest, set + C::weight_col(T, 0, k), b + 2, desc_hi(dK), i32);
                else mma_ts_w<true>(lead, rest, set + C::weight_col(T, 0, k), b + 2, desc_hi(dK), i32);
                mma_ts_w<true>(lead, rest, set + C::weight_col(T, 1, k), b, desc_hi(dK), i32);
                mma_ts_w<true>(lead, rest + 16, set + C::weight_col(T, 2, k), b, desc_hi(dK), i16);
            }
        };
        auto products = [&](int t) -> bool {
            const uint32_t aN = stage_at(t), aW = aN + (C::kNarrow >> 4), set = tb + (t % C::kNSet) * C::kSet;
            const uint32_t turn_col = C::kNAcc == 2 ? (t & 1) * C::kAcc : 0, acc = tb + C::colAcc + turn_col;
            // the first weights (they were formed from this tile's scores: the tile is there)
            if (!mbar_wait(&bars[bWeight + t % C::kNSet], (t / C::kNSet) & 1, abort_flag) ||
                (t >= C::kNAcc && !mbar_wait(&bars[bAccFree + t % C::kNAcc], (t / C::kNAcc - 1) & 1, abort_flag)))
                return false;
            tc_fence_after();
            if (MODE != kDq) {
#pragma unroll
                for (int i = 0; i < 6; ++i)
#pragma unroll
                    for (int k = 0; k < kLT / 16; ++k) {
                        const uint32_t b = desc_lo(dM) + aW + ((part_b(i) * C::kPart) >> 4) + 128 * k;
                        if (i == 0 && k == 0) mma_ts_w<false>(lead, acc, set + C::weight_col(0, part_a(i), k), b, desc_hi(dM), iW);
                        else mma_ts_w<true>(lead, acc, set + C::weight_col(0, part_a(i), k), b, desc_hi(dM), iW);
                    }
            } else {
                narrow(std::integral_constant<int, 0>{}, set, tb + C::colAcc2 + turn_col, tb + C::colRest2, aN, t == 0);
            }
            if (C::kBwd) {
                if (!mbar_wait(&bars[bWeightB + t % C::kNSet], (t / C::kNSet) & 1, abort_flag)) return false;
                tc_fence_after();
                narrow(std::integral_constant<int, 1>{}, set, MODE == kDq ? acc : tb + C::colAcc2,
                       tb + (MODE == kDq ? C::colRest : C::colRest2), aN, t == 0);
            }
            mma_commit_w(lead, &bars[bAccDone + t % C::kNAcc]);
            mma_commit_w(lead, &bars[bSetFree + t % C::kNSet]);
            mma_commit_w(lead, &bars[bEmpty + t % C::kNS]);
            return true;
        };
        if (warp == 12) {
            ok = n == 0 || mbar_wait(&bars[bOwn], 0, abort_flag);
            for (int t = 0; t < n && ok; ++t) ok = scores(t);
        } else {
            for (int t = 0; t < n && ok; ++t) ok = products(t);
        }
    } else if (warp == 13) {
        // ============================================================================ loads
        const uint32_t lead = elect_one();
        const int h = (int)head;
        if (lead && n > 0) {
            mbar_arrive_expect_tx(&bars[bOwn], kOwn * 128 + (C::kBwd ? 3 * C::kOwnPart : 0));
            // (boxes of 64 rows: one map per tensor for both sides)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                tma_load_3d(smem + C::offOwnN + u * (kLT * 128), &tm_own_n, &bars[bOwn], 0, r0 + u * kLT, h);
                if (C::kBwd)
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        tma_load_3d(smem + C::offOwnW + a * C::kOwnPart + u * (kLT * 128), &tm_own_w, &bars[bOwn], a * DV, r0 + u * kLT, h);
            }
        }
        for (int t = 0; t < n && ok; ++t) {
            const int s = t % C::kNS, row = (first + t) * kLT;
            if (t >= C::kNS) ok = mbar_wait(&bars[bEmpty + s], (t / C::kNS - 1) & 1, abort_flag);
            if (!ok || !lead) continue;
            uint8_t* st = smem + C::offStage + s * C::kStage;
            mbar_arrive_expect_tx(&bars[bFull + s], C::kStage + (MODE == kKeys ? 2 * kLT * 4 : 0));
            tma_load_3d(st, &tm_loop_n, &bars[bFull + s], 0, row, h);
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < C::kVB; ++b)
                    tma_load_3d(st + C::kNarrow + a * C::kPart + b * (kLT * 128), &tm_loop_w, &bars[bFull + s], a * p.dvw + 64 * b, row, h);
            if (MODE == kKeys) {
                uint8_t* sst = smem + C::offStats + s * (2 * kLT * 4);
                bulk_load_1d(sst, p.inv + hs + row, kLT * 4, &bars[bFull + s]);
                bulk_load_1d(sst + kLT * 4, p.b + hs + row, kLT * 4, &bars[bFull + s]);
            }
        }
    } else if (warp < 8) {
        // ============================================================================ rows
        const int wg = warp >> 2, row_l = tid & 127, row = r0 + row_l;
        const uint32_t lane_base = (uint32_t)(warp & 3) * 32u;
        const float m_own = MODE == kDq && row < p.L && !p.numerator_only ? p.m[head * (size_t)p.L + row] : 0.f;
        // 1/4, 1/32, 1/16 of scores that are the products of two scaled operands
        const uint64_t k4 = f2(0.25f * kDown2, 0.25f * kDown2), k32 = f2(0.03125f * kDown2 * kDown2, 0.03125f * kDown2 * kDown2);
        const uint64_t k16 = f2(0.0625f * kDown2, 0.0625f * kDown2), one = f2(1.f, 1.f), quarter = f2(0.25f, 0.25f);
        const uint64_t negm = f2(-m_own * kUp, -m_own * kUp), gv_scale = MODE == kDq ? f2(kDown, kDown) : f2(kDown2, kDown2);
        uint64_t den2 = 0, num2 = 0;
        for (int t = C::kBwd ? 0 : wg; t < n; t += C::kBwd ? 1 : 2) {
            const int c0 = (first + t) * kLT, rw = r0 + (int)lane_base;               // the tile's first column, the warp's first row
            const uint32_t set = tmem_addr(tb, lane_base, (t % C::kNSet) * C::kSet);
            const float* st = reinterpret_cast<const float*>(smem + C::offStats) + (t % C::kNS) * (2 * kLT);
            ok = __all_sync(~0u, mbar_wait(&bars[bScore + t % C::kNSet], (t / C::kNSet) & 1, abort_flag));
            if (!ok) break;
            tc_fence_after();
            uint64_t dt = 0, nt = 0;                                   // row sums of this tile
            auto put = [&](int t, int k, const uint32_t (&w)[3][8]) {
                uint32_t x[16];
#pragma unroll
                for (int e = 0; e < 8; ++e) { x[e] = w[0][e]; x[8 + e] = w[1][e]; }
                tmem_st16(set + C::weight_col(t, 0, k), x);
                tmem_st8(set + C::weight_col(t, 2, k), w[2]);
            };
            auto written = [&](int bar) {
                tmem_wait_st();
                tc_fence_before();
                mbar_arrive(&bars[bar]);
            };
            auto products_there = [&] {
                ok = __all_sync(~0u, mbar_wait(&bars[bScoreG + t % C::kNSet], (t / C::kNSet) & 1, abort_flag));
                tc_fence_after();
            };
            // 32 columns of the tile from 32 h on
            auto pass = [&](auto masked_tag, int h) {
                constexpr bool MASKED = decltype(masked_tag)::value;
                uint32_t sr[32], w[3][8];
                tmem_ld32(set + 32 * h, sr);
                tmem_wait_ld();
                auto masked = [&](uint64_t v, int i) {
                    if (!MASKED) return v;
                    const int col = c0 + 32 * h + 2 * i;
                    float lo, hi;
                    unpack2(v, lo, hi);
                    return f2((MODE == kKeys ? row <= col && col < p.L : col <= row) ? lo : 0.f,
                              (MODE == kKeys ? row <= col + 1 && col + 1 < p.L : col + 1 <= row) ? hi : 0.f);
                };
#pragma unroll
                for (int k = 0; k < 2; ++k) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint64_t s = bits2(sr[16 * k + 2 * i], sr[16 * k + 2 * i + 1]);
                        uint64_t wt = MODE == kDq ? fma2(s, k16, quarter) : fma2(s, fma2(s, k32, k4), one);
                        // (past the end 1/D and the mean are anything: masked after the products)
                        if (MODE == kKeys) wt = mul2(wt, *reinterpret_cast<const uint64_t*>(st + 32 * h + 16 * k + 2 * i));
                        wt = masked(wt, 8 * k + i);
                        if (MODE == kFwd) dt = add2(dt, wt);
                        split_pair(wt, w[0][i], w[1][i], w[2][i]);
                    }
                    put(0, 2 * h + k, w);
                }
                if (!C::kBwd) return;
                written(bWeight + t % C::kNSet);
                products_there();
                if (!ok) return;
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    uint32_t gr[16];
                    tmem_ld16(set + kLT + 32 * h + 16 * k, gr);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const uint64_t s = bits2(sr[16 * k + 2 * i], sr[16 * k + 2 * i + 1]), gv = bits2(gr[2 * i], gr[2 * i + 1]);
                        const uint64_t w1 = fma2(s, k16, quarter);
                        uint64_t x;
                        if (MODE == kDq) {
                            const uint64_t wt = masked(fma2(s, fma2(s, k32, k4), one), 8 * k + i);
                            dt = add2(dt, wt);
                            nt = fma2(wt, masked(gv, 8 * k + i), nt);
                            x = mul2(w1, fma2(gv, gv_scale, negm));
                        } else {
                            const float* at = st + 32 * h + 16 * k + 2 * i;
                            x = mul2(mul2(w1, *reinterpret_cast<const uint64_t*>(at)),
                                     fma2(gv, gv_scale, *reinterpret_cast<const uint64_t*>(at + kLT)));
                        }
                        split_pair(masked(x, 8 * k + i), w[0][i], w[1][i], w[2][i]);
                    }
                    put(1, 2 * h + k, w);
                }
            };
            // the warp's rows meet 32 columns: no pair live, some (on the diagonal, or past the sequence's end), or all
#pragma unroll 1
            for (int h = C::kBwd ? wg : 0; h < (C::kBwd ? wg + 1 : 2); ++h) {
                const int cb = c0 + 32 * h;
                const bool dead = MODE == kKeys ? cb < rw : cb > rw;
                const bool some = cb == rw || (MODE == kKeys && cb + 32 > p.L);
                if (dead) {
                    uint32_t z[3][8];
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int e = 0; e < 8; ++e) z[i][e] = 0u;
                    put(0, 2 * h, z);
                    put(0, 2 * h + 1, z);
                    if (C::kBwd) {
                        written(bWeight + t % C::kNSet);
                        products_there();
                        if (!ok) break;
                        put(1, 2 * h, z);
                        put(1, 2 * h + 1, z);
                    }
                } else if (some) {
                    pass(std::true_type{}, h);
                } else {
                    pass(std::false_type{}, h);
                }
            }
            if (!ok) break;
            written(C::kBwd ? bWeightB + t % C::kNSet : bWeight + t % C::kNSet);
            den2 = add2(den2, dt);
            num2 = add2(num2, nt);
        }
        if (MODE != kKeys) {
            float a, b, c, d;
            unpack2(den2, a, b);
            unpack2(num2, c, d);
            s_sum[wg * kOwn + row_l] = make_float2(a + b, c + d);
        }
        ok = workers_all(ok);
    } else {
        // ============================================================================ collectors
        const int row_l = tid & 127, row = r0 + row_l;
        const uint32_t lane_base = (uint32_t)(warp & 3) * 32u;
        // sums over the tiles: Y or dV, and dK; kDq: X, then Y
        constexpr int NA = MODE == kFwd ? DV : MODE == kDq ? 32 : 80;
        uint64_t acc[NA / 2];
#pragma unroll
        for (int i = 0; i < NA / 2; ++i) acc[i] = 0;
        for (int t = 0; t < n; ++t) {
            ok = __all_sync(~0u, mbar_wait(&bars[bAccDone + t % C::kNAcc], (t / C::kNAcc) & 1, abort_flag));
            if (!ok) break;
            tc_fence_after();
            const uint32_t at = tmem_addr(tb, lane_base, C::colAcc + (C::kNAcc == 2 ? (t & 1) * C::kAcc : 0));
#pragma unroll
            for (int h = 0; h < NA / 16; ++h) {
                uint32_t r[16];
                tmem_ld16(at + (MODE == kDq ? C::colAcc2 - C::colAcc : 16) * h, r);
                tmem_wait_ld();
                if (h == NA / 16 - 1) {
                    tc_fence_before();
                    mbar_arrive(&bars[bAccFree + t % C::kNAcc]);
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[8 * h + i] = add2(acc[8 * h + i], bits2(r[2 * i], r[2 * i + 1]));
            }
        }
        ok = workers_all(ok);
        if (ok) {
            float2 sum = make_float2(0.f, 0.f);
            if (MODE != kKeys) {
                const float2 a = s_sum[row_l], b = s_sum[kOwn + row_l];
                sum = make_float2(a.x + b.x, a.y + b.y);
            }
            float x[NA];
#pragma unroll
            for (int i = 0; i < NA / 2; ++i) unpack2(acc[i], x[2 * i], x[2 * i + 1]);
            // the products of smaller parts (32 columns from `col`) on top of x[at ..]
            auto add_rest = [&](int at, uint32_t col) {
                uint32_t r[32];
                tmem_ld32(tmem_addr(tb, lane_base, col), r);
                tmem_wait_ld();
#pragma unroll
                for (int i = 0; i < 16; ++i) x[at + i] += __uint_as_float(r[i]) + __uint_as_float(r[16 + i]);
            };
            if (MODE == kDq && n > 0) {
                add_rest(0, C::colRest);
                add_rest(16, C::colRest2);
            }
            if (MODE == kKeys && n > 0) add_rest(64, C::colRest2);
            if (p.nsplit > 1) {
                // the cluster's sums, through the stages' place (their tiles are used): the first CTA adds the others' to its own
                float* ex = reinterpret_cast<float*>(smem + C::offStage) + row_l;
                if (rank > 0) {
#pragma unroll
                    for (int i = 0; i < NA; ++i) ex[i * kOwn] = x[i];
                    ex[NA * kOwn] = sum.x;
                    ex[(NA + 1) * kOwn] = sum.y;
                }
                cluster_sync();
                for (int r = 1; rank == 0 && r < p.nsplit; ++r) {
                    const float* other = cg::this_cluster().map_shared_rank(ex, r);
#pragma unroll
                    for (int i = 0; i < NA; ++i) x[i] += other[i * kOwn];
                    sum.x += other[NA * kOwn];
                    sum.y += other[(NA + 1) * kOwn];
                }
            }
            const bool mine = rank == 0 && row < p.L;
            auto finite = [&](auto from_tag, auto to_tag, uint64_t chk) {
#pragma unroll
                for (int i = decltype(from_tag)::value; i < decltype(to_tag)::value; i += 2) chk = fma2(f2(x[i], x[i + 1]), 0, chk);
                float a, b;
                unpack2(chk, a, b);
                return a == 0.f && b == 0.f;
            };
            using I0 = std::integral_constant<int, 0>;
            using IW = std::integral_constant<int, MODE == kKeys ? 64 : NA>;
            const bool good = finite(I0{}, IW{}, f2(sum.x * 0.f, sum.y * 0.f));          // 0 x: NaN for an infinite x too
            const bool good_n = MODE == kKeys ? finite(IW{}, std::integral_constant<int, NA>{}, 0) : good;
            if (mine) {
                if (MODE == kDq && good) {
                    const float inv = p.numerator_only ? 1.f : 1.f / (sum.x + kEps);
                    const float mean = p.numerator_only ? 0.f : sum.y * kDown2 * inv;
                    const float c = p.numerator_only ? 0.f : fmaf(p.m[head * (size_t)p.L + row], inv, -mean * inv);
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float o[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) o[e] = fmaf(x[8 * h + e] * kDown2, inv, c * (x[16 + 8 * h + e] * kDown));
                        store8(p.out_n + hn + (size_t)row * kDFeat + 8 * h, o);
                    }
                    p.inv[hs + row] = inv * kUp;
                    p.b[hs + row] = -mean;
                } else if (MODE != kDq && good) {
                    // 1 / D in two parts: as close as a division, two multiply-adds per pair
                    const float d = sum.x + kEps, r = p.numerator_only ? 1.f : 1.f / d, r_lo = p.numerator_only ? 0.f : fmaf(-d, r, 1.f) * r;
                    const uint64_t rr = f2(r, r), rl = f2(r_lo, r_lo), back = MODE == kFwd ? f2(kDown, kDown) : f2(kDown2, kDown2);
                    float* dst = p.out_w + hw + (size_t)row * p.dvw;
#pragma unroll
                    for (int c = 0; c < DV; c += 8) {
                        float o[8];
#pragma unroll
                        for (int e = 0; e < 8; e += 2) {
                            const uint64_t y = mul2(f2(x[c + e], x[c + e + 1]), back);
                            unpack2(MODE == kFwd ? fma2(y, rr, mul2(y, rl)) : y, o[e], o[e + 1]);
                        }
                        if (DV == 64 || c < p.dvw) store8(dst + c, o);
                    }
                }
                if (MODE == kKeys && good_n)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        float o[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) o[e] = x[64 + 8 * h + e] * kDown2;
                        store8(p.out_n + hn + (size_t)row * kDFeat + 8 * h, o);
                    }
            }
            if (__any_sync(~0u, mine && !(good && good_n)))
                plain_rows<MODE>(p, reinterpret_cast<float*>(smem + C::offStage) + (warp - 8) * kPlainFloats, head, row, mine && !good_n,
                                 mine && !good);
        } else if (p.nsplit > 1) {
            cluster_sync();
        }
    }
    if (p.nsplit > 1) {
        if (warp < 8 || warp > 11) cluster_sync();           // the sums are there
        cluster_sync();                                      // and read
    }
    if (!ok && lane == 0) atomicOr(p.err, 1u);
    tc_fence_before();
    __syncthreads();
    if (*abort_flag) {
        for (int i = 0; i < 200; ++i) __nanosleep(1000);     // loads still in flight get time to land
    }
    __syncthreads();
    if (warp == 12) tmem_dealloc(tb, 512);
}

namespace {
struct Maps { CUtensorMap own_n, own_w, loop_n, loop_w; };
template <int DV, int MODE>
based_status launch_quadratic(const Maps& m, QParams p, cudaStream_t stream) {
    using C = QCfg<DV, MODE>;
    if (error_word_ptr(&p.err) != BASED_OK) return BASED_ERR_CUDA;
    {
        static bool configured[64] = {};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BASED_ERR_CUDA;
        std::lock_guard<std::mutex> lock(setup_mutex());
        if (!configured[dev]) {
            if (cudaFuncSetAttribute(quadratic_f32_tc_kernel<DV, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)C::kSmem) != cudaSuccess)
                return BASED_ERR_CUDA;
            configured[dev] = true;
        }
    }
    const long long ctas = (long long)p.heads * ((p.L + kOwn - 1) / kOwn);
    p.by_length = ctas > kSMs;
    // Few own tiles: up to eight CTAs each, as many as fit the chip at once (clusters of eight leave SMs of a GPC unused), two
    // looped tiles each at least (forward and backward, us, of 2 heads L 512 with four: 11.9 / 24.5, with eight 14.2 / 27.2; L 1024
    // 13.2 / 30.1 with four, 17.5 / 56 with one).  Not at d_v 128, where the sums are twice as many: L 500 19 with one, 29 with eight.
    p.nsplit = 1;
    const int tiles = (p.L + kLT - 1) / kLT;
    for (int n = 2; n <= (DV == 64 ? 8 : 1) && ctas * n <= (n == 2 ? 148 : n == 4 ? 128 : 104) && n <= (tiles + 1) / 2; n *= 2) p.nsplit = n;
    const cudaError_t e = launch_ex(quadratic_f32_tc_kernel<DV, MODE>, dim3((unsigned)ctas * p.nsplit), dim3(kNThreads), C::kSmem, p.nsplit, true, stream,
                                    m.own_n, m.own_w, m.loop_n, m.loop_w, p);
    note_launch();
    const based_status st = check_launch("quadratic_f32_tc_kernel");
    return e == cudaSuccess ? st : BASED_ERR_CUDA;
}

// the parts of a call, for as many heads at a time as kPartsBytes hold (one at least)
constexpr size_t kPartsBytes = (size_t)256 << 20;
size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
struct Parts {
    int heads;                                       // per slab
    __nv_bfloat16* n[2];                             // q, k: [heads][L][48]
    __nv_bfloat16* w[2];                             // v, dout: [heads][L][3 d_v]
    float *inv, *b, *m;
    size_t bytes;
};
Parts parts_of(void* ws, int BH, int L, int d_v, bool backward) {
    Parts x{};
    const size_t narrow = (size_t)L * 96, wide = (size_t)L * d_v * 6;
    const size_t per = 2 * narrow + (backward ? 2 : 1) * wide;
    const size_t fit = kPartsBytes / per;
    x.heads = fit < 1 ? 1 : fit < (size_t)BH ? (int)fit : BH;
    const uintptr_t base = reinterpret_cast<uintptr_t>(ws);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const uintptr_t at = base + off;
        off = align256(off + bytes);
        return at;
    };
    for (auto& n : x.n) n = reinterpret_cast<__nv_bfloat16*>(take(x.heads * narrow));
    x.w[0] = reinterpret_cast<__nv_bfloat16*>(take(x.heads * wide));
    if (backward) {
        const size_t stat = (size_t)x.heads * ((L + kLT - 1) / kLT * kLT) * sizeof(float);
        x.w[1] = reinterpret_cast<__nv_bfloat16*>(take(x.heads * wide));
        x.inv = reinterpret_cast<float*>(take(stat));
        x.b = reinterpret_cast<float*>(take(stat));
        x.m = reinterpret_cast<float*>(take(stat));
    }
    x.bytes = off;
    return x;
}
based_status split_parts(const float* const (&src)[4], const Parts& x, int heads, int L, int d_v, bool centres, int dout_H, int h0,
                         cudaStream_t stream) {
    SplitSet s{};
    s.L = L; s.H = dout_H; s.h0 = h0;
    s.m = centres ? x.m : nullptr;
    __nv_bfloat16* const dst[4] = {x.n[0], x.n[1], x.w[0], x.w[1]};
    unsigned end = 0;
    for (int i = 0; i < 4; ++i) {
        s.src[i] = src[i];
        s.dst[i] = dst[i];
        s.pieces[i] = i < 2 ? kDFeat / 8 : d_v / 8;
        s.total[i] = src[i] ? (long long)heads * L * s.pieces[i] : 0;
        end += (unsigned)((s.total[i] + kSplitBlock - 1) / kSplitBlock);
        s.end[i] = end;
    }
    // (a dependent launch takes the host 1.7 us, a plain one 1.9)
    const cudaError_t e = launch_ex(split_parts_kernel, dim3(end), dim3(256), 0, 1, true, stream, s);
    note_launch();
    const based_status st = check_launch("split_parts_kernel");
    return e == cudaSuccess ? st : BASED_ERR_CUDA;
}
bool narrow_map(CUtensorMap* m, const void* base, int heads, int L) {
    return make_rows_map_bf16(m, base, heads, L, 3 * kDFeat, 64, kLT, CU_TENSOR_MAP_SWIZZLE_128B);
}
bool wide_map(CUtensorMap* m, const void* base, int heads, int L, int d_v) {
    return make_rows_map_bf16(m, base, heads, L, 3 * d_v, 64, kLT, CU_TENSOR_MAP_SWIZZLE_128B);
}
}  // namespace

size_t quadratic_f32_workspace_bytes(int BH, int L, int d_v, bool backward) {
    // Forward (us, this / the chunked kernel of prefill_f32.cu, whose time grows with L alone; that one has two or three CTAs per head
    // for 38 to 74 heads).  Short: d_v 64 L 25 to 32 7.2 / 8.5 up to 128 heads, 8.8 / 8.6 with 148, 24 / 21 with 500, then L 33 24 /
    // 30; d_v 128 L 32 10.3 / 9.0, L 33 10.3 / 13.4, with 47 or 64 heads 11.4 / 10.9 at L 33 and 41, 10.7 / 10.8 at L 48.
    // Between: L 1024 13.4 / 20.8 with 2 heads, 27 / 72 with 32, 45 / 146 with 32 at d_v 128.  Long: L 4096 483 / 622 with 64 heads
    // (898 / 924 at d_v 128), L 3840 690 / 746 with 96, at d_v 128 1250 / 1497, but 1030 / 866 with 74 there; L 3000 616 / 683 with
    // 128, L 2816 1077 / 1062 with 256, L 2432 840 / 917; L 8192 99 / 154 with 2, 404 / 393 with 16.
    if (!backward) {
        const bool two = d_v != 64 && BH > 37 && BH <= 74;
        const int from = two ? 49 : d_v != 64 || BH > 128 ? 33 : 25;
        const int to = BH <= 64 ? 4096 : two ? 3072 : BH <= 96 ? 3840 : BH <= 128 ? 2816 : 2432;
        if (L < from || L > to) return 0;
    } else {
        // Backward, against backward_f32.cu (quadratic too, d_v 64): L 1 to 64 13.6 to 17 / 14.5 to 18 up to 74 heads; with more the
        // 128 own rows of a CTA are half empty and that one's 64 are not: L 64 18.2 / 17.9 with 80 heads, 65 / 50 with 500, L 32 41 /
        // 34 with 300.  From L 65 on 55 / 69 (300 heads, L 80), L 1024 30 / 45 with 2, 80 / 268 with 32.  That one gives a cluster a
        // tile of 64 and a CTA one tile of its loop where heads are few: L 193 to 256 with up to 8 heads 21 to 25 / 20 to 21, with 16
        // 25 / 30; L 449 to 512 with one 24 / 19.6, with two 24 / 26 to 28.
        if (d_v != 64 || (L <= kLT && BH > 74) || (L > 192 && L <= 256 && BH <= 8) || (L > 448 && L <= 512 && BH == 1)) return 0;
    }
    return parts_of(nullptr, BH, L, d_v, backward).bytes;
}

based_status launch_quadratic_forward_f32(const float* q, const float* k, const float* v, float* out, void* ws, int BH, int L,
                                          int d_v, int numerator_only, cudaStream_t stream) {
    const Parts x = parts_of(ws, BH, L, d_v, false);
    const size_t hn = (size_t)L * kDFeat, hw = (size_t)L * d_v;
    for (int h0 = 0; h0 < BH; h0 += x.heads) {
        QParams p{};
        p.heads = BH - h0 < x.heads ? BH - h0 : x.heads;
        p.own_n = q + h0 * hn; p.loop_n = k + h0 * hn; p.loop_w = v + h0 * hw; p.out_w = out + h0 * hw;
        p.L = L; p.dvw = d_v; p.numerator_only = numerator_only;
        const float* const src[4] = {p.own_n, p.loop_n, p.loop_w, nullptr};
        based_status st = split_parts(src, x, p.heads, L, d_v, false, 0, 0, stream);
        if (st != BASED_OK) return st;
        Maps m;
        if (!narrow_map(&m.own_n, x.n[0], p.heads, L) || !narrow_map(&m.loop_n, x.n[1], p.heads, L) ||
            !wide_map(&m.loop_w, x.w[0], p.heads, L, d_v))
            return BASED_ERR_CUDA;
        m.own_w = m.own_n;
        st = d_v == 64 ? launch_quadratic<64, kFwd>(m, p, stream) : launch_quadratic<128, kFwd>(m, p, stream);
        if (st != BASED_OK) return st;
    }
    return BASED_OK;
}

based_status launch_quadratic_backward_f32(const float* q, const float* k, const float* v, const float* g, int dout_H, float* dq,
                                           float* dk, float* dv, void* ws, int BH, int L, int numerator_only, cudaStream_t stream) {
    constexpr int DV = 64;
    const Parts x = parts_of(ws, BH, L, DV, true);
    const size_t hn = (size_t)L * kDFeat, hw = (size_t)L * DV;
    for (int h0 = 0; h0 < BH; h0 += x.heads) {
        QParams p{};
        p.heads = BH - h0 < x.heads ? BH - h0 : x.heads;
        p.L = L; p.dvw = DV; p.numerator_only = numerator_only;
        p.inv = x.inv; p.b = x.b; p.m = x.m; p.pitch = (L + kLT - 1) / kLT * kLT;
        p.dout_H = dout_H; p.dout_h0 = h0;
        const float* const src[4] = {q + h0 * hn, k + h0 * hn, v + h0 * hw, dout_H ? g : g + h0 * hw};
        based_status st = split_parts(src, x, p.heads, L, DV, !numerator_only, dout_H, h0, stream);
        if (st != BASED_OK) return st;
        Maps m;
        if (!narrow_map(&m.own_n, x.n[0], p.heads, L) || !wide_map(&m.own_w, x.w[1], p.heads, L, DV) ||
            !narrow_map(&m.loop_n, x.n[1], p.heads, L) || !wide_map(&m.loop_w, x.w[0], p.heads, L, DV))
            return BASED_ERR_CUDA;
        p.own_n = src[0]; p.own_w = src[3]; p.loop_n = src[1]; p.loop_w = src[2];
        p.out_n = dq + h0 * hn;
        if ((st = launch_quadratic<DV, kDq>(m, p, stream)) != BASED_OK) return st;
        std::swap(m.own_n, m.loop_n);
        std::swap(m.own_w, m.loop_w);
        p.own_n = src[1]; p.own_w = src[2]; p.loop_n = src[0]; p.loop_w = src[3];
        p.out_n = dk + h0 * hn; p.out_w = dv + h0 * hw;
        if ((st = launch_quadratic<DV, kKeys>(m, p, stream)) != BASED_OK) return st;
    }
    return BASED_OK;
}

}  // namespace based
