// based_prefill for fp32 io (d' = 16): causal Taylor linear attention with fp32 FMAs.  In chunked form, the sequence of a head
// spread over the CTAs of one thread-block cluster; where there is less to do (f32_short_rows) in definition form, further down.
//
// One bf16 or tf32 operand per fp32 value cannot meet fp32's tolerance (three bf16 parts can: quadratic_f32_tc.cu, training's
// forward pass, in definition form and without a state), so the contractions are register-tiled products on the fp32 pipe (two-wide fma.rn.f32x2), fed from shared memory.  One CTA holds 64 value columns of one sequence
// segment; the cluster's CTAs are the segments of a head in order (and, above 64 columns, its column groups):
//   1. every segment sums its own state  S_seg = sum_j psi(k_j) v_j^T  (153 features, one per unordered pair) and z_seg,
//      and leaves it in shared memory;
//   2. the cluster turns these sums, on top of the caller's state, into running sums in place: every CTA takes a share of
//      the elements through all segments' shared memory and writes that share of the final state (no scratch in global
//      memory, one launch);
//   3. chunks of 64 tokens: out = (psi(Q) S + P V) / (psi(Q) z + rowsum P), P = (1 + s/4 + s^2/32)[j <= i] with
//      s = q.k, then, unless it is the segment's last chunk, S += psi(K)^T V, z += sum psi(K).
// With one segment there is no step 1 and 2 and every chunk of step 3 updates the state.
// Every operand lies along its product's summation index (f32_tiles.cuh).  Outputs: a warp owns 16 query rows and a slice of
// the features; four slices' groups of 16 rows make a full chunk's eight warps two slices, a chunk of at most 32 (16) tokens
// has four (eight), and the slices' sums meet in shared memory.
// Bound: issue slots and latency (per full chunk and SM 28 k cycles, the FMA pipe busy in 12.6 k of them; 11 k instructions per
// scheduler, 6.8 k of them multiply-adds); at few heads the chain of steps.  Against one CTA per head that walked the tokens
// one by one: B1 H2 L256 d_v64 190 -> 15 us, B2 H16 L1024 d_v64 660 -> 74.  An earlier form with the operands row by row
// along the summation index (even and odd terms in one two-wide FMA) took 22 and 92: twice the shared-memory passes, and
// chunks of 16 tokens used a quarter of the warps' rows.
#include <cooperative_groups.h>
#include <math.h>

#include "common.cuh"
#include "f32_tiles.cuh"

namespace based {

namespace {
namespace cg = cooperative_groups;

constexpr int kTok = 64;           // tokens per chunk
constexpr int kNT = 256;
constexpr int kMaxSeg = 16;        // CTAs of the largest cluster
constexpr int kRowT = 68;          // row pitch of tiles with 64 tokens per row
constexpr int kRowX = 20;          // row pitch of k rows: 16 values, then 1 (0 past the end)
constexpr int kWarpRows = 16;
// the definition form (prefill_f32_short_kernel)
constexpr int kGroup = 32;         // keys or tokens of a warp's turn
constexpr int kPsiCols = 20;       // features of a state CTA, or of a warp for a continued call's read-out
constexpr int kStateCtas = kFeatRows / kPsiCols;

struct F32Smem {
    float psi[kFeat * kRowT];      // in turn: the warps' P^T [32 keys][16 rows] each, psi(Q)^T [156][68], the slices'
                                   // sums, psi(K) [64][160]
    float st[kFeat * 64];          // state [156 features][64 columns]
    float z[kFeatRows];
    float v[kTok * 64];            // V of the chunk
    float xq[(kDFeat + 1) * kRowT], xk[kDFeat * kRowT];      // transposed; xq: a row of ones behind
    float kr[kTok * kRowX];        // k rows as they lie
    float den[kTok];
    FeatTab tab;
};
static_assert(2 * (sizeof(F32Smem) + 1024) <= 228 * 1024, "two CTAs per SM");
static_assert(kTok * kFeatRows <= kFeat * kRowT, "psi(K) fits");

// The head's state in the caller's arrays, by symmetric feature f (order of based_decode_step_sym): the row itself, or the
// rows (m, n) and (n, m) of a full state.
struct AbiState {
    float* kv;                     // the head's first row, first column of this CTA
    float* z;
    int pitch;
    // A continued full state gets what the call adds to the sum of the rows (m, n) and (n, m), not the sum folded back into
    // both: 1 / sqrt 2 there and back is 3.4e-8 short of a half in fp32, in the same direction on every call (300 short pieces
    // left the pair rows 9e-6 low).  So a row that nothing is added to stays bit for bit, and the rows may differ.
    bool sym, add;
    static __device__ __forceinline__ float added(float x, float before) { return x == before ? 0.f : x - before; }   // (inf: nothing)
    __device__ __forceinline__ void rows(const FeatTab& tab, int f, int& a, int& b) const {
        a = b = f;
        if (sym || f <= kDFeat) return;
        const int m = tab.mn[f] & 255, n = tab.mn[f] >> 8;
        a = 1 + kDFeat + m * kDFeat + n;
        b = 1 + kDFeat + n * kDFeat + m;
    }
    static __device__ __forceinline__ float fold(float x, float y, bool two) { return two ? __fmul_rn(x + y, kRsqrt2) : x; }
    __device__ __forceinline__ float4 kv_get(const FeatTab& tab, int f, int c) const {
        int a, b;
        rows(tab, f, a, b);
        const float4 x = *reinterpret_cast<const float4*>(kv + (size_t)a * pitch + c);
        const float4 y = *reinterpret_cast<const float4*>(kv + (size_t)b * pitch + c);
        const bool two = a != b;
        return make_float4(fold(x.x, y.x, two), fold(x.y, y.y, two), fold(x.z, y.z, two), fold(x.w, y.w, two));
    }
    __device__ __forceinline__ void kv_put(const FeatTab& tab, int f, int c, float4 x, bool pair) const {
        int a, b;
        rows(tab, f, a, b);
        float4* pa = reinterpret_cast<float4*>(kv + (size_t)a * pitch + c);
        float4* pb = reinterpret_cast<float4*>(kv + (size_t)b * pitch + c);
        if (!pair) {
            *pa = x;
            return;
        }
        float4 u = make_float4(0.f, 0.f, 0.f, 0.f), w = u;
        if (add) {
            u = *pa;
            w = *pb;
            x = make_float4(added(x.x, fold(u.x, w.x, true)), added(x.y, fold(u.y, w.y, true)), added(x.z, fold(u.z, w.z, true)),
                            added(x.w, fold(u.w, w.w, true)));
        }
        *pa = make_float4(fmaf(x.x, kRsqrt2, u.x), fmaf(x.y, kRsqrt2, u.y), fmaf(x.z, kRsqrt2, u.z), fmaf(x.w, kRsqrt2, u.w));
        *pb = make_float4(fmaf(x.x, kRsqrt2, w.x), fmaf(x.y, kRsqrt2, w.y), fmaf(x.z, kRsqrt2, w.z), fmaf(x.w, kRsqrt2, w.w));
    }
    __device__ __forceinline__ void kv_put(const FeatTab& tab, int f, int c, float4 x) const {
        int a, b;
        rows(tab, f, a, b);
        kv_put(tab, f, c, x, a != b);
    }
    // The call's own sum x of feature f added to its row or rows, which hold u and w (kv_rows, z_rows)
    __device__ __forceinline__ void kv_rows(const FeatTab& tab, int f, int c, float4& u, float4& w) const {
        int a, b;
        rows(tab, f, a, b);
        u = *reinterpret_cast<const float4*>(kv + (size_t)a * pitch + c);
        w = *reinterpret_cast<const float4*>(kv + (size_t)b * pitch + c);
    }
    __device__ __forceinline__ void kv_add(const FeatTab& tab, int f, int c, float4 x, float4 u, float4 w) const {
        int a, b;
        rows(tab, f, a, b);
        const float s = a != b ? kRsqrt2 : 1.f;
        *reinterpret_cast<float4*>(kv + (size_t)a * pitch + c) = make_float4(fmaf(x.x, s, u.x), fmaf(x.y, s, u.y), fmaf(x.z, s, u.z), fmaf(x.w, s, u.w));
        if (a != b)
            *reinterpret_cast<float4*>(kv + (size_t)b * pitch + c) = make_float4(fmaf(x.x, s, w.x), fmaf(x.y, s, w.y), fmaf(x.z, s, w.z), fmaf(x.w, s, w.w));
    }
    __device__ __forceinline__ void z_rows(const FeatTab& tab, int f, float& u, float& w) const {
        int a, b;
        rows(tab, f, a, b);
        u = z[a];
        w = z[b];
    }
    __device__ __forceinline__ void z_add(const FeatTab& tab, int f, float x, float u, float w) const {
        int a, b;
        rows(tab, f, a, b);
        const float s = a != b ? kRsqrt2 : 1.f;
        z[a] = fmaf(x, s, u);
        if (a != b) z[b] = fmaf(x, s, w);
    }
    __device__ __forceinline__ float z_get(const FeatTab& tab, int f) const {
        int a, b;
        rows(tab, f, a, b);
        return fold(z[a], z[b], a != b);
    }
    __device__ __forceinline__ void z_put(const FeatTab& tab, int f, float x) const {
        int a, b;
        rows(tab, f, a, b);
        if (a == b) {
            z[a] = x;
            return;
        }
        const float u = add ? z[a] : 0.f, w = add ? z[b] : 0.f;
        if (add) x = added(x, fold(u, w, true));
        z[a] = fmaf(x, kRsqrt2, u);
        z[b] = fmaf(x, kRsqrt2, w);
    }
};

// up to 64 rows of 16 values, transposed -> [16][68]; rows past nt are zero.  rows: as they lie too, element 16 1 on real rows
__device__ __forceinline__ void load_x(float* dst, float* rows, const float* __restrict__ src, int nt, int tid) {
    const int t = tid >> 2, p = tid & 3;
    const bool live = t < nt;
    const float4 x = live ? __ldg(reinterpret_cast<const float4*>(src + (size_t)t * kDFeat) + p) : make_float4(0.f, 0.f, 0.f, 0.f);
    dst[(4 * p + 0) * kRowT + t] = x.x;
    dst[(4 * p + 1) * kRowT + t] = x.y;
    dst[(4 * p + 2) * kRowT + t] = x.z;
    dst[(4 * p + 3) * kRowT + t] = x.w;
    if (rows) {
        *reinterpret_cast<float4*>(&rows[t * kRowX + 4 * p]) = x;
        if (p == 0) rows[t * kRowX + kDFeat] = live ? 1.f : 0.f;
    }
}
// 64 tokens x 64 columns of a row-major array; tokens past nt and columns past ncol (a multiple of 4) are zero.  Whether all
// of this thread's values are finite.
__device__ __forceinline__ bool load_v(float* dst, const float* __restrict__ src, int pitch, int ncol, int nt, int tid) {
    float4 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int t = (tid >> 4) + 16 * i, c = (tid & 15) * 4;
        x[i] = t < nt && c < ncol ? __ldg(reinterpret_cast<const float4*>(src + (size_t)t * pitch + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(&dst[((tid >> 4) + 16 * i) * 64 + (tid & 15) * 4]) = x[i];
    float zero = 0.f;                                // 0 x: NaN for an infinite x too
#pragma unroll
    for (int i = 0; i < 4; ++i) zero = fmaf(x[i].x, 0.f, fmaf(x[i].y, 0.f, fmaf(x[i].z, 0.f, fmaf(x[i].w, 0.f, zero))));
    return zero == 0.f;
}

// acc (rows in pairs: row0 + {0..3, 8..11}, columns 4 co + j) += sum_{k < n} a[k][row] b[k][column]
__device__ __forceinline__ void tile_product(float2 (&acc)[4][4], const float* a, int pa, const float* b, int pb, int n) {
#pragma unroll 4
    for (int k = 0; k < n; ++k, a += pa, b += pb) {
        const float4 x0 = lds4(a), x1 = lds4(a + 8), y = lds4(b);
        const float ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            fma_pair(acc[0][j], x0.x, x0.y, ys[j]);
            fma_pair(acc[1][j], x0.z, x0.w, ys[j]);
            fma_pair(acc[2][j], x1.x, x1.y, ys[j]);
            fma_pair(acc[3][j], x1.z, x1.w, ys[j]);
        }
    }
}
// state tile of a thread, features 8 fg + 2 i + {0, 1} (i < 4) and 128 + 2 fg + {0, 1} (i = 4), columns 4 cg + j:
// += sum_{t < nt} psi(K)[t][feature] V[t][column]
__device__ __forceinline__ void state_product(float2 (&acc)[5][4], const float* psi, const float* v, int nt, int fg, int cg) {
    const float *a = psi + 8 * fg, *a2 = psi + 128 + 2 * fg, *b = v + 4 * cg;
#pragma unroll 2
    for (int t = 0; t < nt; ++t, a += kFeatRows, a2 += kFeatRows, b += 64) {
        const float4 x0 = lds4(a), x1 = lds4(a + 4), y = lds4(b);
        const float2 x2 = *reinterpret_cast<const float2*>(a2);
        const float ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            fma_pair(acc[0][j], x0.x, x0.y, ys[j]);
            fma_pair(acc[1][j], x0.z, x0.w, ys[j]);
            fma_pair(acc[2][j], x1.x, x1.y, ys[j]);
            fma_pair(acc[3][j], x1.z, x1.w, ys[j]);
            fma_pair(acc[4][j], x2.x, x2.y, ys[j]);
        }
    }
}

// The in-chunk product where V holds infinities or NaN: a masked weight times one would be NaN in rows that do not see the
// key, so such pairs are left out instead of multiplied by zero.  row0: the thread's first row relative to the first key.
// (What it costs a call on finite values is 0 to 1.5 %, measured: B2 H16 L1024 d_v64 72.9 -> 73.7 us, 148 heads L640 139.4
// -> 139.5.  Out of line, or as a pass over the stored outputs, it cost as much or more.)
__device__ __forceinline__ void causal_product(float2 (&acc)[4][4], const float* a, const float* b, int n, int row0) {
#pragma unroll 1
    for (int k = 0; k < n; ++k, a += kWarpRows, b += 64) {
        const float4 y = lds4(b);
        const float ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (k > row0 + (i >> 2) * 8 + (i & 3)) continue;
            const float w = a[(i >> 2) * 8 + (i & 3)];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float& x = i & 1 ? acc[i >> 1][j].y : acc[i >> 1][j].x;
                x = fmaf(w, ys[j], x);
            }
        }
    }
}

// Outputs of a chunk of nt <= 16 NR tokens; ends with a barrier.  Warp w: rows 16 (w % NR), slice w / NR of 8 / NR.
// state_ready is called before the state is read.  finite: all of V is.
template <int NR, class F>
__device__ __forceinline__ void chunk_outputs(F32Smem& s, float* __restrict__ o, int d_v, int ncol, int nt, bool numerator_only,
                                              bool finite, int tid, F&& state_ready) {
    constexpr int KS = 8 / NR;
    const int warp = tid >> 5, lane = tid & 31, ro = lane & 1, co = lane >> 1;
    const int rg = warp % NR, ks = warp / NR, row0 = rg * kWarpRows + ro * 4;
    float2 acc[4][4];
    float den[8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 8; ++i) den[i] = 0.f;
    // in-chunk part: 32 keys per slice (a chunk of more than 32 tokens has two slices of keys), weights in the warp's own
    // place, [key][16 rows]
    if (32 * ks < nt) {
        float* pw = s.psi + warp * (32 * kWarpRows);
        float2 p[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i][0] = p[i][1] = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int k = 0; k < kDFeat; ++k) {
            const float4 x0 = lds4(&s.xq[k * kRowT + row0]), x1 = lds4(&s.xq[k * kRowT + row0 + 8]);
            const float2 y = *reinterpret_cast<const float2*>(&s.xk[k * kRowT + 32 * ks + 2 * co]);
            fma_pair(p[0][0], x0.x, x0.y, y.x); fma_pair(p[0][1], x0.x, x0.y, y.y);
            fma_pair(p[1][0], x0.z, x0.w, y.x); fma_pair(p[1][1], x0.z, x0.w, y.y);
            fma_pair(p[2][0], x1.x, x1.y, y.x); fma_pair(p[2][1], x1.x, x1.y, y.y);
            fma_pair(p[3][0], x1.z, x1.w, y.x); fma_pair(p[3][1], x1.z, x1.w, y.y);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float x = i & 1 ? p[i >> 1][j].y : p[i >> 1][j].x;
                const int row = row0 + (i >> 2) * 8 + (i & 3), key = 32 * ks + 2 * co + j;
                w[i] = key <= row ? fmaf(x, fmaf(x, 0.03125f, 0.25f), 1.0f) : 0.f;
                den[i] += w[i];
            }
            float* at = pw + (2 * co + j) * kWarpRows + ro * 4;
            *reinterpret_cast<float4*>(at) = make_float4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<float4*>(at + 8) = make_float4(w[4], w[5], w[6], w[7]);
        }
        __syncwarp();
        // no key behind the warp's last row counts
        const int n = min(32, max(0, min(nt, (rg + 1) * kWarpRows) - 32 * ks));
        if (finite) tile_product(acc, pw + ro * 4, kWarpRows, s.v + 32 * ks * 64 + 4 * co, 64, n);
        else causal_product(acc, pw + ro * 4, s.v + 32 * ks * 64 + 4 * co, n, row0 - 32 * ks);
    }
    __syncthreads();                                 // P is read: psi(Q)^T takes its place
    for (int e = tid; e < kFeat * (NR * 4); e += kNT) {
        // four tokens of a feature; consecutive lanes: consecutive features
        const int t = e / kFeat * 4, f = e % kFeat;
        const float4 a = lds4(&s.xq[(s.tab.mn[f] & 255) * kRowT + t]), b = lds4(&s.xq[(s.tab.mn[f] >> 8) * kRowT + t]);
        const float c = s.tab.scale[f];
        *reinterpret_cast<float4*>(&s.psi[f * kRowT + t]) = make_float4(c * a.x * b.x, c * a.y * b.y, c * a.z * b.z, c * a.w * b.w);
    }
    state_ready();
    __syncthreads();
    const int f0 = ks * kFeat / KS, f1 = (ks + 1) * kFeat / KS;
    tile_product(acc, s.psi + f0 * kRowT + row0, kRowT, s.st + f0 * 64 + 4 * co, 64, f1 - f0);
    for (int f = f0 + co; f < f1; f += 16) {
        const float4 x0 = lds4(&s.psi[f * kRowT + row0]), x1 = lds4(&s.psi[f * kRowT + row0 + 8]);
        const float zf = s.z[f];
        den[0] = fmaf(x0.x, zf, den[0]); den[1] = fmaf(x0.y, zf, den[1]); den[2] = fmaf(x0.z, zf, den[2]); den[3] = fmaf(x0.w, zf, den[3]);
        den[4] = fmaf(x1.x, zf, den[4]); den[5] = fmaf(x1.y, zf, den[5]); den[6] = fmaf(x1.z, zf, den[6]); den[7] = fmaf(x1.w, zf, den[7]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int x = 2; x < 32; x <<= 1) den[i] += __shfl_xor_sync(0xffffffffu, den[i], x);
    __syncthreads();                                 // psi(Q)^T is read: the slices' sums take its place
    float* red = s.psi + (ks - 1) * (NR * kWarpRows * 64);
    float* red_den = s.psi + (KS - 1) * (NR * kWarpRows * 64);
    if (ks > 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = row0 + (i >> 2) * 8 + (i & 3);
            *reinterpret_cast<float4*>(&red[row * 64 + 4 * co]) =
                i & 1 ? make_float4(acc[i >> 1][0].y, acc[i >> 1][1].y, acc[i >> 1][2].y, acc[i >> 1][3].y)
                      : make_float4(acc[i >> 1][0].x, acc[i >> 1][1].x, acc[i >> 1][2].x, acc[i >> 1][3].x);
            if (co == 0) red_den[(ks - 1) * (NR * kWarpRows) + row] = den[i];
        }
    }
    __syncthreads();
    if (ks == 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int row = row0 + (i >> 2) * 8 + (i & 3);
            float4 x = i & 1 ? make_float4(acc[i >> 1][0].y, acc[i >> 1][1].y, acc[i >> 1][2].y, acc[i >> 1][3].y)
                             : make_float4(acc[i >> 1][0].x, acc[i >> 1][1].x, acc[i >> 1][2].x, acc[i >> 1][3].x);
            float d = den[i];
#pragma unroll
            for (int r = 0; r < KS - 1; ++r) {
                const float4 y = lds4(&s.psi[r * (NR * kWarpRows * 64) + row * 64 + 4 * co]);
                x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
                d += red_den[r * (NR * kWarpRows) + row];
            }
            if (row < nt && 4 * co < ncol) {
                d = numerator_only ? 1.f : d + kEps;
                *reinterpret_cast<float4*>(&o[(size_t)row * d_v + 4 * co]) = make_float4(x.x / d, x.y / d, x.z / d, x.w / d);
            }
        }
    }
    __syncthreads();                                 // the slices' sums are read
}
}  // namespace

__global__ void __launch_bounds__(kNT, 2)
    prefill_f32_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                       float* __restrict__ out, float* kv, float* z, int L, int seg, int d_v, int ncol, int flags) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    F32Smem& s = *reinterpret_cast<F32Smem*>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int nseg = gridDim.x, rank = blockIdx.x;   // the cluster: all segments and column groups of a head
    const int cluster_row = blockIdx.z * nseg;
    const size_t head = blockIdx.y;
    const int col0 = blockIdx.z * ncol;
    const int tid = threadIdx.x, lane = tid & 31;
    const int fg = (tid >> 5) * 2 + (lane & 1), cgr = lane >> 1;     // state tile (state_product)
    const int t_begin = min(rank * seg, L), t_end = min(t_begin + seg, L);
    const bool cont = (flags & BASED_STATE_CONTINUE) != 0, numerator_only = (flags & BASED_NUMERATOR_ONLY) != 0;
    AbiState abi;
    abi.sym = (flags & BASED_STATE_SYM) != 0;
    abi.add = cont && !abi.sym;
    abi.pitch = d_v;
    abi.kv = kv + head * (size_t)(abi.sym ? kDSym : kD) * d_v + col0;
    abi.z = z + head * (size_t)(abi.sym ? kDSym : kD);

    const float* qh = q + head * (size_t)L * kDFeat;
    const float* kh = k + head * (size_t)L * kDFeat;
    const float* vh = v + head * (size_t)L * d_v + col0;
    float* oh = out + head * (size_t)L * d_v + col0;

    fill_feat_tab(s.tab, tid);
    if (tid < kRowT) s.xq[kDFeat * kRowT + tid] = 1.f;
    __syncthreads();

    float2 acc[5][4];
    auto clear = [&] {
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
    };
    // a chunk's contribution to the state tile; psi(K) is left in place for z
    auto chunk_state = [&](int nt) {
        // a lane's five features of every eighth token
#pragma unroll
        for (int i = 0; i < kFeatRows / 32; ++i) {
            const int f = lane + 32 * i;
            const float *xm = s.kr + (s.tab.mn[f] & 255), *xn = s.kr + (s.tab.mn[f] >> 8);
            const float c = s.tab.scale[f];
#pragma unroll
            for (int u = 0; u < kTok / 8; ++u) {
                const int t = (tid >> 5) + 8 * u;
                if (8 * u < nt) s.psi[t * kFeatRows + f] = c * xm[t * kRowX] * xn[t * kRowX];
            }
        }
        __syncthreads();
        state_product(acc, s.psi, s.v, nt, fg, cgr);
    };
    auto chunk_z = [&](int nt) {                     // thread f < 160
        float a[4] = {0.f, 0.f, 0.f, 0.f};           // (rows past nt up to the next eight are zero)
        for (int t = 0; t < nt; t += 8)
#pragma unroll
            for (int u = 0; u < 8; ++u) a[u & 3] += s.psi[(t + u) * kFeatRows + tid];
        return (a[0] + a[1]) + (a[2] + a[3]);
    };
    // the state tile's elements: feature, columns 4 cgr .. + 3
    auto each_row = [&](auto fn) {
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int f = (i < 4 ? 8 * fg + 2 * i : 128 + 2 * fg) + h;
                if (f < kFeat)
                    fn(f, h ? make_float4(acc[i][0].y, acc[i][1].y, acc[i][2].y, acc[i][3].y)
                            : make_float4(acc[i][0].x, acc[i][1].x, acc[i][2].x, acc[i][3].x));
            }
    };
    bool summed = true;                              // the running sums are complete
    if (nseg > 1) {
        // ---- step 1: this segment's own state (the last one's is needed for the final state only)
        clear();
        float zsum = 0.f;                            // thread f < 160: z of feature f
        const float zc = cont && rank == 0 && tid < kDSym ? abi.z_get(s.tab, tid) : 0.f;
        if (rank < nseg - 1 || kv != nullptr) {
            for (int t0 = t_begin; t0 < t_end; t0 += kTok) {
                const int nt = min(kTok, t_end - t0);
                load_x(s.xk, s.kr, kh + (size_t)t0 * kDFeat, nt, tid);
                load_v(s.v, vh + (size_t)t0 * d_v, d_v, ncol, nt, tid);
                __syncthreads();
                chunk_state(nt);
                if (tid < kFeatRows) zsum += chunk_z(nt);
                __syncthreads();
            }
        }
        each_row([&](int f, float4 x) { *reinterpret_cast<float4*>(&s.st[f * 64 + 4 * cgr]) = x; });
        if (tid < kFeatRows) s.z[tid] = zsum;
        cluster.sync();

        // ---- step 2: running sums over the segments, four columns of a feature per thread
        for (int e = rank * kNT + tid; e < kFeat * 16; e += nseg * kNT) {
            const int f = e >> 4, c = (e & 15) * 4;
            float4* mine = reinterpret_cast<float4*>(&s.st[f * 64 + c]);
            float4 x[kMaxSeg];
#pragma unroll
            for (int r = 0; r < kMaxSeg; ++r)
                if (r < nseg) x[r] = *cluster.map_shared_rank(mine, cluster_row + r);
            const bool real = f < kDSym && c < ncol;
            float4 run = cont && real ? abi.kv_get(s.tab, f, c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int r = 0; r < kMaxSeg; ++r)
                if (r < nseg) {
                    *cluster.map_shared_rank(mine, cluster_row + r) = run;
                    run.x += x[r].x; run.y += x[r].y; run.z += x[r].z; run.w += x[r].w;
                }
            if (kv != nullptr && real) abi.kv_put(s.tab, f, c, run);
        }
        if (rank == 0 && tid < kFeatRows) {
            float x[kMaxSeg], run = zc;
#pragma unroll
            for (int r = 0; r < kMaxSeg; ++r)
                if (r < nseg) x[r] = *cluster.map_shared_rank(&s.z[tid], cluster_row + r);
#pragma unroll
            for (int r = 0; r < kMaxSeg; ++r)
                if (r < nseg) {
                    *cluster.map_shared_rank(&s.z[tid], cluster_row + r) = run;
                    run += x[r];
                }
            if (z != nullptr && blockIdx.z == 0 && tid < kDSym) abi.z_put(s.tab, tid, run);
        }
        // the wait for the other CTAs' share comes when the first chunk needs the state: behind its loads, weights and psi(Q)
        // (B1 H2 L256 15.3 -> 14.7 us, B2 H16 L1024 74.7 -> 71.9; one load of a one-chunk segment for steps 1 and 3 gives 0.2 us
        // more there and costs 3 % at B4 H16 L2048)
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        summed = false;
    } else {
        for (int e = tid; e < kFeat * 16; e += kNT) {
            const int f = e >> 4, c = (e & 15) * 4;
            *reinterpret_cast<float4*>(&s.st[f * 64 + c]) =
                cont && f < kDSym && c < ncol ? abi.kv_get(s.tab, f, c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (tid < kFeatRows) s.z[tid] = cont && tid < kDSym ? abi.z_get(s.tab, tid) : 0.f;
        // column group 0 writes the K-state that the other one reads
        if (cont && gridDim.z > 1) cluster.sync();
    }

    // ---- step 3: outputs, chunk by chunk
    auto state_ready = [&] {
        if (!summed) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        summed = true;
    };
    for (int t0 = t_begin; t0 < t_end; t0 += kTok) {
        const int nt = min(kTok, t_end - t0);
        load_x(s.xq, nullptr, qh + (size_t)t0 * kDFeat, nt, tid);
        load_x(s.xk, s.kr, kh + (size_t)t0 * kDFeat, nt, tid);
        const bool finite = __syncthreads_and(load_v(s.v, vh + (size_t)t0 * d_v, d_v, ncol, nt, tid));
        float* o = oh + (size_t)t0 * d_v;
        if (nt > 32) chunk_outputs<4>(s, o, d_v, ncol, nt, numerator_only, finite, tid, state_ready);
        else if (nt > 16) chunk_outputs<2>(s, o, d_v, ncol, nt, numerator_only, finite, tid, state_ready);
        else chunk_outputs<1>(s, o, d_v, ncol, nt, numerator_only, finite, tid, state_ready);
        if (t0 + kTok >= t_end && (nseg > 1 || kv == nullptr)) break;   // nobody reads the state after this chunk
        clear();
        chunk_state(nt);
        each_row([&](int f, float4 x) {
            float4* p = reinterpret_cast<float4*>(&s.st[f * 64 + 4 * cgr]);
            float4 y = *p;
            y.x += x.x; y.y += x.y; y.z += x.z; y.w += x.w;
            *p = y;
        });
        if (tid < kFeatRows) s.z[tid] += chunk_z(nt);
        __syncthreads();
    }

    state_ready();                                   // (a segment without tokens)
    if (nseg == 1 && kv != nullptr) {
        for (int e = tid; e < kDSym * 16; e += kNT) {
            const int f = e >> 4, c = (e & 15) * 4;
            if (c < ncol) abi.kv_put(s.tab, f, c, lds4(&s.st[f * 64 + c]));
        }
        if (blockIdx.z == 0 && tid < kDSym) abi.z_put(s.tab, tid, s.z[tid]);
    }
}

namespace {
// whole groups of 16 tokens, so that every segment but the last ends on a tile edge of the products
int f32_segment_tokens(int L, int nseg) { return ((L + nseg - 1) / nseg + 15) / 16 * 16; }
// Segments per head (the cluster holds all segments of both column groups, at most 16 CTAs), by a time model fitted on
// B200, in us: outputs of a full chunk 9.3 (a chunk of up to 32 / 16 tokens 6.8 / 6), a state update 4.9 (3.8 / 3.5), 3 for
// launch and ramps, 3 + 0.1 n for the running sums of n segments; two CTAs on an SM 1.8 times one, more in proportion.
// Clusters of 8 and 16 CTAs leave SMs of a GPC unused: about 104 and 96 CTAs fit one per SM, and many waves take 1.15 and
// 1.4 times as long.  More segments shorten the chain of chunks but every chunk then updates a state twice (its segment's
// own sums, then the running state).  Measured with 1 / 2 / 4 / 8 / 16 segments: B1 H2 L256 d_v64 60 / 39 / 20 / 17 / 16,
// B2 H16 L1024 d_v64 229 / 154 / 78 / 75 / 80, B8 H16 L512 d_v64 117 / 130 / 121 / 118 / 201, B1 H16 L700 d_v64 159 / 111 /
// 57 / 55 / 47.  The same whether the state is asked for or not: so are the outputs.
int f32_segments(int BH, int L, int nz, double* time) {
    int best = 1;
    double best_t = 1e30;
    for (int n = 1; n * nz <= kMaxSeg; n *= 2) {
        const int seg = f32_segment_tokens(L, n), full = seg / kTok, rest = seg % kTok;
        const double outs = full * 9.3 + (rest == 0 ? 0.0 : rest <= 16 ? 6.0 : rest <= 32 ? 6.8 : 9.3);
        const double ups = full * 4.9 + (rest == 0 ? 0.0 : rest <= 16 ? 3.5 : rest <= 32 ? 3.8 : 4.9);
        const double last = rest == 0 ? 4.9 : rest <= 16 ? 3.5 : rest <= 32 ? 3.8 : 4.9;
        const int cl = n * nz;
        const double ctas = (double)BH * cl, fit = cl <= 4 ? 148 : cl == 8 ? 104 : 96;
        const double many = ctas / 148 * (cl <= 4 ? 1.0 : cl == 8 ? 1.15 : 1.4);
        const double load = ctas <= fit ? 1.0 : many > 1.8 ? many : 1.8;
        const double t = load * (outs + (n > 1 ? 2 * ups - last : ups)) + 3.0 + (n > 1 ? 3.0 + 0.1 * n : 0.0);
        if (t < best_t) { best_t = t; best = n; }
    }
    *time = best_t;
    return best;
}
// 16-row groups per CTA of the definition form, 1 or 2, or 0 where the chunked kernel (time: its model's us) is the faster.  A
// time model of the same kind, fitted where the two are close (within 5 % there; further away it is up to 25 % off, on the right
// side): a CTA's loop of g groups, or all CTAs' groups over the chip, whichever is longer, the state's CTAs among them; a
// continued call has the state's features as more keys and a second launch, and there one group of rows is always the better.
// The chunked kernel's model is 7 % high on these shapes; where the two are within 12 % of each other it keeps the call (a
// continued call of one segment per head reads the state in 4 us more than the model says).
// Measured, us, chunked / one / two groups, with a new state: B1 H2 L256 15.1 / 6.2 / 7.9, L1024 21.2 / 16.3 / 23.2, H8 L600
// 30.0 / 20.8 / 24.5, L1024 31.8 / 38.0 / 38.3, H64 L33 16.5 / 12.9 / 10.3, L200 31.9 / 30.1 / 28.0, L256 32.0 / 35.2 / 32.7;
// continued: H2 L256 15.7 / 11.6, L1024 21.9 / 19.4, H64 L16 17.2 / 15.0, L128 22.5 / 30.2.  The same whether a new state is
// asked for or not: so are the outputs.
int f32_short_rows(int BH, int L, int nz, bool continued, double time) {
    if (L > 2048) return 0;
    auto keys_loop = [](int keys, int slices) { return ((keys + kGroup - 1) / kGroup + slices - 1) / slices; };
    auto longer = [](double a, double b) { return cbrt(a * a * a + b * b * b); };
    const double per_sm = (double)BH * nz / kSMs, state = per_sm * kStateCtas * keys_loop(L, 8);
    double best_t = time * (0.88 / 1.07);
    int best = 0;
    for (int nr = 1; nr <= (continued ? 1 : 2); ++nr) {
        const int rows = nr * kWarpRows, tiles = (L + rows - 1) / rows;
        int sum = 0;
        for (int i = 1; i <= tiles; ++i) sum += keys_loop(i * rows < L ? i * rows : L, 8 / nr);
        const int most = keys_loop(L, 8 / nr);
        const double t = nr == 2 ? 4.8 + longer(2.2 * most, per_sm * (2.0 * tiles + 3.3 * sum) + state)
                         : continued ? 3.8 + longer(3.7 * most, per_sm * (3.6 * tiles + 2.7 * sum)) + longer(3.5, 1.4 * state + 3.7 * per_sm)
                                     : 3.8 + longer(3.7 * most, per_sm * (0.9 * tiles + 2.7 * sum) + 1.4 * state);
        if (t < best_t) { best_t = t; best = nr; }
    }
    return best;
}
}  // namespace

// ---- the definition form: few heads of a short sequence ------------------------------------------------------------------
// The chunked kernel's chain (a segment's own state, the cluster's running sums, then the outputs) takes 16 us however little
// there is to do, on a few CTAs per head.  Here every CTA starts from the inputs and none waits for another:
//   outputs: a CTA has 16 NR query rows and all keys up to them, its warps 16 rows each and every 8 / NR-th group of 32 keys;
//   state:   a CTA has 20 features of a head and all tokens, its warps every eighth group of 32.
// A warp loads its groups' k and v rows itself (cp.async; the other warps and the SM's other CTA cover its wait), so that nothing in
// the loop is waited for by the whole CTA; the warps' sums meet in shared memory at the end.
// A continued call reads the caller's state as 153 more keys, 20 to a warp (weights psi(q), values the state's rows), and adds
// to it in a second launch of the same kernel that sums beside the first one and waits for its end before it writes.
// Bound: the chain launch -> first loads -> one to a few groups a warp (1.3 k issue cycles each) -> sums; with many rows the
// fp32 pipe.  B1 H2 L256 d_v64 with state 15.1 -> 6.2 us, continued 15.7 -> 11.6; H16 L400 30.5 -> 21.1.  With a second stage
// per warp, one CTA per SM, 5.8 and 23.6: the other CTA hides more.
struct ShortSmem {
    struct Stage {
        float k[kGroup * kRowX];   // element 16 of a row is 1
        float v[kGroup * 64];
    } st[8];
    float w[8][kGroup * kPsiCols]; // a warp's weights [key][16 rows], or psi(k) [token][20 features]
    float xq[(kDFeat + 1) * 68];   // q rows, transposed; a row of ones behind
    FeatTab tab;
};
static_assert(2 * (sizeof(ShortSmem) + 1024) <= 228 * 1024, "two CTAs per SM");

__device__ __forceinline__ void cp_async16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
template <int NR>
__global__ void __launch_bounds__(kNT, 2)
    prefill_f32_short_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                             float* __restrict__ out, float* kv, float* z, int L, int d_v, int ncol, int flags, int state_ctas,
                             int beside) {
    constexpr int KS = 8 / NR;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ShortSmem& s = *reinterpret_cast<ShortSmem*>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, ro = lane & 1, co = lane >> 1;
    const size_t head = blockIdx.y;
    const int col0 = blockIdx.z * ncol;
    const bool cont = (flags & BASED_STATE_CONTINUE) != 0, numerator_only = (flags & BASED_NUMERATOR_ONLY) != 0;
    AbiState abi;
    abi.sym = (flags & BASED_STATE_SYM) != 0;
    abi.add = cont && !abi.sym;
    abi.pitch = d_v;
    abi.kv = kv + head * (size_t)(abi.sym ? kDSym : kD) * d_v + col0;
    abi.z = z + head * (size_t)(abi.sym ? kDSym : kD);
    const float* kh = k + head * (size_t)L * kDFeat;
    const float* vh = v + head * (size_t)L * d_v + col0;

    fill_feat_tab(s.tab, tid);
    if (tid < 68) s.xq[kDFeat * 68 + tid] = 1.f;
    s.st[warp].k[lane * kRowX + kDFeat] = 1.f;
    // beside: the launch ahead is this call's own, which lets this one start when the call's inputs are there
    if (!beside) asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    ShortSmem::Stage& d = s.st[warp];
    auto load = [&](int g) {
        const int t0 = g * kGroup, nt = min(kGroup, L - t0);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = (lane >> 2) + 8 * i, c = (lane & 3) * 4;
            if (t < nt) cp_async16(&d.k[t * kRowX + c], kh + (size_t)(t0 + t) * kDFeat + c);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int t = (lane >> 4) + 2 * i, c = (lane & 15) * 4;
            if (t < nt && c < ncol) cp_async16(&d.v[t * 64 + c], vh + (size_t)(t0 + t) * d_v + c);
        }
    };
    // groups first, first + step .. below n
    auto each_group = [&](int first, int step, int n, auto use) {
        for (int g = first; g < n; g += step) {
            load(g);
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            use(g, d);
            __syncwarp();
        }
    };
    float* pw = s.w[warp];
    float* red = s.st[0].k;        // the warps' sums, over the stages

    if ((int)blockIdx.x < state_ctas) {
        // ==================================================================== state: features f0 .. f0 + 19
        const int f0 = blockIdx.x * kPsiCols;
        float2 sum[5][4];          // of sixteen tokens' sums each: no long chain of additions
        float zs = 0.f;            // lane < 20: z of feature f0 + lane
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) sum[i][j] = make_float2(0.f, 0.f);
        __syncthreads();           // the table
        each_group(warp, 8, (L + kGroup - 1) / kGroup, [&](int g, const ShortSmem::Stage& st) {
            const int nt = min(kGroup, L - g * kGroup);
            const float* x = st.k + lane * kRowX;
            if (lane < nt) {
#pragma unroll
                for (int i = 0; i < kPsiCols; i += 4) {
                    float y[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t mn = s.tab.mn[f0 + i + j];
                        y[j] = s.tab.scale[f0 + i + j] * x[mn & 255] * x[mn >> 8];
                    }
                    *reinterpret_cast<float4*>(&pw[lane * kPsiCols + i]) = make_float4(y[0], y[1], y[2], y[3]);
                }
            }
            __syncwarp();
            const float *a = pw + 8 * ro, *a2 = pw + 16 + 2 * ro, *b = st.v + 4 * co;
#pragma unroll 1
            for (int t0 = 0; t0 < nt; t0 += 16) {
                float2 acc[5][4];
#pragma unroll
                for (int i = 0; i < 5; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 4
                for (int t = t0; t < min(t0 + 16, nt); ++t, a += kPsiCols, a2 += kPsiCols, b += 64) {
                    const float4 x0 = lds4(a), x1 = lds4(a + 4), y = lds4(b);
                    const float2 x2 = *reinterpret_cast<const float2*>(a2);
                    const float ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        fma_pair(acc[0][j], x0.x, x0.y, ys[j]);
                        fma_pair(acc[1][j], x0.z, x0.w, ys[j]);
                        fma_pair(acc[2][j], x1.x, x1.y, ys[j]);
                        fma_pair(acc[3][j], x1.z, x1.w, ys[j]);
                        fma_pair(acc[4][j], x2.x, x2.y, ys[j]);
                    }
                }
#pragma unroll
                for (int i = 0; i < 5; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) { sum[i][j].x += acc[i][j].x; sum[i][j].y += acc[i][j].y; }
            }
            if (lane < kPsiCols) {
                float y[4] = {0.f, 0.f, 0.f, 0.f};
                int t = 0;
                for (; t + 4 <= nt; t += 4)
#pragma unroll
                    for (int u = 0; u < 4; ++u) y[u] += pw[(t + u) * kPsiCols + lane];
                for (; t < nt; ++t) y[0] += pw[t * kPsiCols + lane];
                zs += (y[0] + y[1]) + (y[2] + y[3]);
            }
        });
        __syncthreads();           // the stages are read
#pragma unroll
        for (int i = 0; i < 5; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int f = (i < 4 ? 8 * ro + 2 * i : 16 + 2 * ro) + h;
                *reinterpret_cast<float4*>(&red[(warp * kPsiCols + f) * 64 + 4 * co]) =
                    h ? make_float4(sum[i][0].y, sum[i][1].y, sum[i][2].y, sum[i][3].y)
                      : make_float4(sum[i][0].x, sum[i][1].x, sum[i][2].x, sum[i][3].x);
            }
        float* red_z = red + 8 * kPsiCols * 64;
        if (lane < kPsiCols) red_z[warp * kPsiCols + lane] = zs;
        // what the caller's state holds, requested before the wait for the outputs' launch, which reads it too
        constexpr int kMine = (kPsiCols * 16 + kNT - 1) / kNT;
        float4 ra[kMine], rb[kMine];
        float za = 0.f, zb = 0.f;
        const int zf = f0 + tid;
        const bool z_mine = blockIdx.z == 0 && tid < kPsiCols && zf < kDSym;
        auto mine = [&](int i, int& f, int& c) {
            const int e = tid + i * kNT;
            f = f0 + (e >> 4);
            c = (e & 15) * 4;
            return e < kPsiCols * 16 && f < kDSym && c < ncol;
        };
        if (cont) {
            int f, c;
#pragma unroll
            for (int i = 0; i < kMine; ++i)
                if (mine(i, f, c)) abi.kv_rows(s.tab, f, c, ra[i], rb[i]);
            if (z_mine) abi.z_rows(s.tab, zf, za, zb);
        }
        if (beside) asm volatile("griddepcontrol.wait;" ::: "memory");
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kMine; ++i) {
            int f, c;
            if (!mine(i, f, c)) continue;
            const float* r = &red[(f - f0) * 64 + c];
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int w = 0; w < 8; w += 2) {             // pairs first
                const float4 y = lds4(r + w * kPsiCols * 64), u = lds4(r + (w + 1) * kPsiCols * 64);
                x.x += y.x + u.x; x.y += y.y + u.y; x.z += y.z + u.z; x.w += y.w + u.w;
            }
            if (cont) abi.kv_add(s.tab, f, c, x, ra[i], rb[i]);
            else abi.kv_put(s.tab, f, c, x);
        }
        if (z_mine) {
            float x = 0.f;
#pragma unroll
            for (int w = 0; w < 8; w += 2) x += red_z[w * kPsiCols + tid] + red_z[(w + 1) * kPsiCols + tid];
            if (cont) abi.z_add(s.tab, zf, x, za, zb);
            else abi.z_put(s.tab, zf, x);
        }
        return;
    }

    // ======================================================================== outputs: rows r0 .. r0 + 16 NR - 1
    const int tiles = gridDim.x - state_ctas, r0 = (tiles - 1 - ((int)blockIdx.x - state_ctas)) * (kWarpRows * NR);    // the longest first
    const int rg = warp % NR, ks = warp / NR, row0 = rg * kWarpRows + ro * 4;
    const int end = min(L, r0 + (rg + 1) * kWarpRows);       // keys of the warp's rows
    const float* qh = q + head * (size_t)L * kDFeat;
    if (tid < NR * kWarpRows * 4) {
        const int t = tid >> 2, c = (tid & 3) * 4;
        const float4 x = r0 + t < L ? *reinterpret_cast<const float4*>(qh + (size_t)(r0 + t) * kDFeat + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        s.xq[(c + 0) * 68 + t] = x.x;
        s.xq[(c + 1) * 68 + t] = x.y;
        s.xq[(c + 2) * 68 + t] = x.z;
        s.xq[(c + 3) * 68 + t] = x.w;
    }
    if (cont) {                    // on its way to L2 while the keys are worked on
        const int rows = abi.sym ? kDSym : kD, lines = (ncol * 4 + 127) / 128;
        for (int e = tid; e < rows * lines; e += kNT)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(abi.kv + (size_t)(e / lines) * d_v + (e % lines) * 32));
    }
    __syncthreads();
    float2 acc[4][4];
    float den[8];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 8; ++i) den[i] = 0.f;
    each_group(ks, KS, r0 + rg * kWarpRows < L ? (end + kGroup - 1) / kGroup : 0, [&](int g, const ShortSmem::Stage& st) {
        const int key0 = g * kGroup, n = min(kGroup, end - key0);
        float2 p[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i) p[i][0] = p[i][1] = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < kDFeat; c += 4) {
            const float4 ya = lds4(&st.k[(2 * co) * kRowX + c]), yb = lds4(&st.k[(2 * co + 1) * kRowX + c]);
            const float y0[4] = {ya.x, ya.y, ya.z, ya.w}, y1[4] = {yb.x, yb.y, yb.z, yb.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float4 x0 = lds4(&s.xq[(c + e) * 68 + row0]), x1 = lds4(&s.xq[(c + e) * 68 + row0 + 8]);
                fma_pair(p[0][0], x0.x, x0.y, y0[e]); fma_pair(p[0][1], x0.x, x0.y, y1[e]);
                fma_pair(p[1][0], x0.z, x0.w, y0[e]); fma_pair(p[1][1], x0.z, x0.w, y1[e]);
                fma_pair(p[2][0], x1.x, x1.y, y0[e]); fma_pair(p[2][1], x1.x, x1.y, y1[e]);
                fma_pair(p[3][0], x1.z, x1.w, y0[e]); fma_pair(p[3][1], x1.z, x1.w, y1[e]);
            }
        }
        // (a key past the warp's rows, loaded or not, counts for none of them)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float w[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float x = i & 1 ? p[i >> 1][j].y : p[i >> 1][j].x;
                const int row = r0 + row0 + (i >> 2) * 8 + (i & 3), key = key0 + 2 * co + j;
                w[i] = key <= row && 2 * co + j < n ? fmaf(x, fmaf(x, 0.03125f, 0.25f), 1.0f) : 0.f;
                den[i] += w[i];
            }
            float* at = pw + (2 * co + j) * kWarpRows + ro * 4;
            *reinterpret_cast<float4*>(at) = make_float4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<float4*>(at + 8) = make_float4(w[4], w[5], w[6], w[7]);
        }
        // where some pairs are masked, a weight of zero must not meet an infinite value
        bool finite = true;
        if (key0 + n - 1 > r0 + rg * kWarpRows) {
            float zero = 0.f;
            for (int e = lane; e < n * 16; e += 32) {
                const float4 x = lds4(&st.v[e * 4]);
                if ((e & 15) * 4 < ncol) zero = fmaf(x.x, 0.f, fmaf(x.y, 0.f, fmaf(x.z, 0.f, fmaf(x.w, 0.f, zero))));
            }
            finite = __all_sync(~0u, zero == 0.f);
        }
        __syncwarp();
        if (finite) tile_product(acc, pw + ro * 4, kWarpRows, st.v + 4 * co, 64, n);
        else causal_product(acc, pw + ro * 4, st.v + 4 * co, n, r0 + row0 - key0);
    });
    if (cont) {
        // The caller's state, 20 features at a time, weights psi(q) [feature][16 rows].  Behind the keys: its terms are the large
        // ones, and what is added to them is rounded at their size.
        for (int f0 = ks * kPsiCols; f0 < kDSym; f0 += KS * kPsiCols) {
            float* sv = d.v;
            const int n = min(kPsiCols, kDSym - f0);
#pragma unroll
            for (int i = 0; i < kPsiCols / 2; ++i) {
                const int f = (lane >> 4) + 2 * i, c = (lane & 15) * 4;
                if (f < n && c < ncol) *reinterpret_cast<float4*>(&sv[f * 64 + c]) = abi.kv_get(s.tab, f0 + f, c);
            }
            if (lane < n) d.k[lane * kRowX + kDFeat + 1] = abi.z_get(s.tab, f0 + lane);
            for (int e = lane; e < n * kWarpRows; e += 32) {
                const int f = f0 + (e >> 4), r = rg * kWarpRows + (e & 15);
                const uint32_t mn = s.tab.mn[f];
                pw[e] = s.tab.scale[f] * s.xq[(mn & 255) * 68 + r] * s.xq[(mn >> 8) * 68 + r];
            }
            __syncwarp();
            // ten features' sums at a time, so that few additions are rounded at the whole sum's size (error against 64 bits, one chain behind
            // the keys and the slices one after the other / this, L188 1.6e-7 / 1.25e-7, the chunked kernel's 1.4e-7; 8 heads L16 10.3 / 10.5 us)
#pragma unroll 1
            for (int h = 0; h < n; h += kPsiCols / 2) {
                float2 part[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) part[i][j] = make_float2(0.f, 0.f);
                tile_product(part, pw + h * kWarpRows + ro * 4, kWarpRows, sv + h * 64 + 4 * co, 64, min(kPsiCols / 2, n - h));
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 4; ++j) { acc[i][j].x += part[i][j].x; acc[i][j].y += part[i][j].y; }
            }
            for (int f = co; f < n; f += 16) {
                const float zf = d.k[f * kRowX + kDFeat + 1];
#pragma unroll
                for (int i = 0; i < 8; ++i) den[i] = fmaf(pw[f * kWarpRows + ro * 4 + (i >> 2) * 8 + (i & 3)], zf, den[i]);
            }
            __syncwarp();
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int x = 2; x < 32; x <<= 1) den[i] += __shfl_xor_sync(0xffffffffu, den[i], x);
    __syncthreads();               // the stages are read
    constexpr int kRows = NR * kWarpRows;
    float* red_den = red + KS * kRows * 64;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int row = row0 + (i >> 2) * 8 + (i & 3);
        *reinterpret_cast<float4*>(&red[(ks * kRows + row) * 64 + 4 * co]) =
            i & 1 ? make_float4(acc[i >> 1][0].y, acc[i >> 1][1].y, acc[i >> 1][2].y, acc[i >> 1][3].y)
                  : make_float4(acc[i >> 1][0].x, acc[i >> 1][1].x, acc[i >> 1][2].x, acc[i >> 1][3].x);
        if (co == 0) red_den[ks * kRows + row] = den[i];
    }
    __syncthreads();
    for (int e = tid; e < kRows * 16; e += kNT) {
        const int row = e >> 4, c = (e & 15) * 4;
        if (r0 + row >= L || c >= ncol) continue;
        // two, then four, then all
        auto slices = [&](int w) {
            const float4 x = lds4(&red[(w * kRows + row) * 64 + c]), y = lds4(&red[((w + 1) * kRows + row) * 64 + c]);
            return make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w);
        };
        auto slices_den = [&](int w) { return red_den[w * kRows + row] + red_den[(w + 1) * kRows + row]; };
        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
        float d = 0.f;
#pragma unroll
        for (int w = 0; w < KS; w += 4) {
            const float4 y = slices(w), u = slices(w + 2);
            x.x += y.x + u.x; x.y += y.y + u.y; x.z += y.z + u.z; x.w += y.w + u.w;
            d += slices_den(w) + slices_den(w + 2);
        }
        d = numerator_only ? 1.f : d + kEps;
        *reinterpret_cast<float4*>(&out[(head * L + r0 + row) * (size_t)d_v + col0 + c]) = make_float4(x.x / d, x.y / d, x.z / d, x.w / d);
    }
}

namespace {
template <int NR>
based_status launch_short(const float* q, const float* k, const float* v, float* out, float* kv, float* z, int BH, int L, int d_v,
                          int nz, int flags, cudaStream_t stream) {
    auto kern = prefill_f32_short_kernel<NR>;
    {
        static bool configured[64] = {};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BASED_ERR_CUDA;
        std::lock_guard<std::mutex> lock(setup_mutex());
        if (!configured[dev]) {
            if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ShortSmem)) != cudaSuccess)
                return BASED_ERR_CUDA;
            configured[dev] = true;
        }
    }
    const int tiles = (L + NR * kWarpRows - 1) / (NR * kWarpRows);
    // a continued call's state is written by a launch of its own
    const bool two = (flags & BASED_STATE_CONTINUE) != 0;
    for (int pass = 0; pass < (two ? 2 : 1); ++pass) {
        const int state_ctas = two ? pass * kStateCtas : kv ? kStateCtas : 0;
        const cudaError_t e = launch_ex(kern, dim3(state_ctas + (pass == 0 ? tiles : 0), BH, nz), dim3(kNT), sizeof(ShortSmem), 1, true,
                                        stream, q, k, v, out, kv, z, L, d_v, d_v / nz, flags, state_ctas, pass);
        note_launch();
        const based_status st = check_launch("prefill_f32_short_kernel");
        if (e != cudaSuccess || st != BASED_OK) return BASED_ERR_CUDA;
    }
    return BASED_OK;
}
}  // namespace

based_status launch_prefill_f32(const void* q, const void* k, const void* v, void* out, float* kv, float* z, int BH,
                                int L, int d_v, int flags, cudaStream_t stream) {
    const int nz = d_v > 64 ? 2 : 1, ncol = d_v / nz;        // 64 or (d_v 112) 56 columns per CTA
    double time = 0.0;
    const int nseg = f32_segments(BH, L, nz, &time), seg = f32_segment_tokens(L, nseg);
    const bool continued = (flags & BASED_STATE_CONTINUE) != 0;
    if (const int nr = f32_short_rows(BH, L, nz, continued, continued && nseg == 1 ? time + 4.0 : time)) {
        auto in = [](const void* p) { return static_cast<const float*>(p); };
        float* o = static_cast<float*>(out);
        return nr == 1 ? launch_short<1>(in(q), in(k), in(v), o, kv, z, BH, L, d_v, nz, flags, stream)
                       : launch_short<2>(in(q), in(k), in(v), o, kv, z, BH, L, d_v, nz, flags, stream);
    }
    {
        static bool configured[64] = {};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BASED_ERR_CUDA;
        std::lock_guard<std::mutex> lock(setup_mutex());
        if (!configured[dev]) {
            if (cudaFuncSetAttribute(prefill_f32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(F32Smem)) != cudaSuccess ||
                cudaFuncSetAttribute(prefill_f32_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
                return BASED_ERR_CUDA;
            configured[dev] = true;
        }
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(nseg, BH, nz);
    cfg.blockDim = dim3(kNT);
    cfg.dynamicSmemBytes = sizeof(F32Smem);
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = nseg;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = nz;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(
        &cfg, prefill_f32_kernel, static_cast<const float*>(q), static_cast<const float*>(k), static_cast<const float*>(v),
        static_cast<float*>(out), kv, z, L, seg, d_v, ncol, flags);
    note_launch();
    const based_status st = check_launch("prefill_f32_kernel");
    return e == cudaSuccess ? st : BASED_ERR_CUDA;
}

}  // namespace based
