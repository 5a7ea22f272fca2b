// based_prefill_backward for fp32 io (d' = 16): gradients of the causal Taylor linear attention (definition form, left-hand
// side of Eq. (2) of Sec. 4.1).  The paper gives no backward algorithm; this is the chain rule on the definition, evaluated
// tile by tile in the quadratic ("attention") form with fp32 FMAs.  d_v 112 and 128, and d_v 64 where operands split into bf16
// parts for the tensor cores (quadratic_f32_tc.cu) are not the faster or have no scratch:
//
//   y_i = N_i / D_i,  N_i = sum_{j<=i} w_ij v_j,  D_i = sum_{j<=i} w_ij + eps,  w_ij = 1 + s/4 + s^2/32,
//   s = q_i.k_j;  with G_i the gradient of the loss with respect to y_i:
//   a_i = G_i / D_i,  b_i = -(G_i.y_i) / D_i = -(G_i.N_i) / D_i^2,  ds_ij = (a_i.v_j + b_i)(1/4 + s_ij/16),
//   dq_i = sum_{j<=i} ds_ij k_j,   dk_j = sum_{i>=j} ds_ij q_i,   dv_j = sum_{i>=j} w_ij a_i.
//
// Two launches over 64 x 64 tiles of (own, looped) rows, one CTA of 128 threads per own tile:
//   dq       own = queries, loops over the key tiles j <= i.  Row statistics and dq in one sweep: with m_i = G_i.v_i,
//            X_i = sum_j w'_ij (G_i.v_j - m_i) k_j and Y_i = sum_j w'_ij k_j, w' = 1/4 + s/16,
//            dq_i = X_i / D_i + (m_i / D_i + b_i) Y_i needs neither D_i nor b_i while the keys are swept (any m_i gives the
//            same sum; this one is exact for the first row, where the two terms of ds cancel).
//   dk, dv   own = keys, loops over the query tiles i >= j.
// A thread holds 8 x 4 pairs of s and G.v in registers, a warp 16 own rows; what a warp needs of its own weights for the
// products over the looped rows (X, Y, dk, dv) goes through shared memory of its own, in tiles laid out along the
// summation index.  Lanes 2n and 2n + 1 differ in the own rows only: a 128-bit load whose neighbouring lanes share an
// address costs two passes, four otherwise.  Few tiles: the CTAs of a cluster share one own tile's loop, and their sums
// are added through distributed shared memory in a fixed order.
// Measured against three sweeps of 4 x 8 pairs per thread on scalar shared-memory loads: B2 H16 L1024 d_v64 1050 -> 424 us,
// B1 H2 L1024 d_v64 50 us with eight CTAs per own tile; 424 -> 294 us with the longest loops of all heads first and one
// weight at a time in shared memory, 275 with two products per instruction (B4 H16 L2048 2090 -> 1823, of which the FMA
// pipe needs 1050).  Bound: issue slots and latency of two CTAs of four warps per SM.  Three CTAs (168 registers, the weights
// in the looped tile's place) 328 to 350 us: their spills and the extra barrier cost what the third CTA hides.
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"
#include "f32_tiles.cuh"

namespace based {

namespace {
namespace cg = cooperative_groups;

constexpr int kT = 64;             // tile edge
constexpr int kBT = 128;           // threads: 4 warps of 16 own rows
constexpr int kP = 68;             // row pitch of tiles with 64 entries per row
constexpr int kMaxSplit = 8;       // CTAs of a cluster that share an own tile

template <int DV, bool KEYS>
struct BwdSmem {
    static constexpr int kCols = (DV + 63) / 64 * 64;
    static constexpr int kWide = kCols + 4;
    float an[kDFeat * kP];         // own q (keys pass: k), transposed [16][68]
    float aw[DV * kP];             // own dout (v), transposed [DV][68]
    float bn[kDFeat * kP];         // looped k (q), transposed
    float bw[DV * kP];             // looped v (dout), transposed
    float rn[kT * kDFeat];         // looped k (q) as it lies, row t at place of(t)
    float rw[KEYS ? kT * kWide : 4];    // looped dout as it lies
    float p[4][kT * 16];           // per warp: a weight of (looped row at place of(t), own row)
    float2 st[kT];                 // keys pass: (1 / D, b) of the looped queries
    float m[kT];
};
// place of looped row t where four consecutive rows belong to one thread: spreads those over the banks
__device__ __forceinline__ int place_of(int t) { return (t & 3) * 16 + (t >> 2); }

// 64 rows of W values (a multiple of 16) of a row-major array (LIES: `pitch` apart), transposed -> [W][68]; rows from nt on are zero.
// nat: the rows as they lie too, at pitch natp (of: at place_of(t))
template <int W, bool LIES = false>
__device__ __forceinline__ void load_tile(float* dst, float* nat, int natp, bool of, const float* __restrict__ src, int nt,
                                          int warp, int lane, size_t pitch = W) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int t = (lane & 7) + 8 * warp + 32 * h;
        float4 x[W / 16];
#pragma unroll
        for (int i = 0; i < W / 16; ++i) {
            x[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (t < nt) x[i] = __ldg(reinterpret_cast<const float4*>(src + (size_t)t * (LIES ? pitch : W)) + (lane >> 3) + 4 * i);
        }
#pragma unroll
        for (int i = 0; i < W / 16; ++i) {
            const int c = 4 * ((lane >> 3) + 4 * i);
            dst[(c + 0) * kP + t] = x[i].x;
            dst[(c + 1) * kP + t] = x[i].y;
            dst[(c + 2) * kP + t] = x[i].z;
            dst[(c + 3) * kP + t] = x[i].w;
            if (nat) *reinterpret_cast<float4*>(&nat[(of ? place_of(t) : t) * natp + c]) = x[i];
        }
    }
}

// s[i / 2][j], element i % 2, += sum_k a[k][row i] b[k][4 co + j]
template <int K>
__device__ __forceinline__ void pair_product(float2 (&s)[4][4], const float* a, const float* b) {
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float4 x0 = lds4(a + k * kP), x1 = lds4(a + k * kP + 8), y = lds4(b + k * kP);
        const float ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            fma_pair(s[0][j], x0.x, x0.y, ys[j]);
            fma_pair(s[1][j], x0.z, x0.w, ys[j]);
            fma_pair(s[2][j], x1.x, x1.y, ys[j]);
            fma_pair(s[3][j], x1.z, x1.w, ys[j]);
        }
    }
}
// acc[i][d / 2], element d % 2, += sum over this lane group's 16 looped rows of p[row][4 rg + i] n[row][8 dg + d]
__device__ __forceinline__ void narrow_product(float2 (&acc)[4][4], const float* p, const float* n, int ks, int rg, int dg) {
#pragma unroll 4
    for (int u = 0; u < 16; ++u) {
        const int r = u * 4 + ks;
        const float4 x = lds4(p + r * 16 + rg * 4), y0 = lds4(n + r * 16 + dg * 8), y1 = lds4(n + r * 16 + dg * 8 + 4);
        const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            fma_pair(acc[i][0], y0.x, y0.y, xs[i]);
            fma_pair(acc[i][1], y0.z, y0.w, xs[i]);
            fma_pair(acc[i][2], y1.x, y1.y, xs[i]);
            fma_pair(acc[i][3], y1.z, y1.w, xs[i]);
        }
    }
}
// one weight of a thread's own rows and looped row 4 co + j
__device__ __forceinline__ void store_weight(float* p, const float (&a)[8], int j, int co, int ro) {
    float* at = p + (j * 16 + co) * 16 + ro * 4;                     // place_of(4 co + j)
    *reinterpret_cast<float4*>(at) = make_float4(a[0], a[1], a[2], a[3]);
    *reinterpret_cast<float4*>(at + 8) = make_float4(a[4], a[5], a[6], a[7]);
}
// sums over the four lane groups ks (lane bits 3, 4)
__device__ __forceinline__ void narrow_reduce(float2 (&acc)[4][4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int d = 0; d < 4; ++d)
#pragma unroll
            for (int o = 8; o < 32; o <<= 1) {
                acc[i][d].x += __shfl_xor_sync(0xffffffffu, acc[i][d].x, o);
                acc[i][d].y += __shfl_xor_sync(0xffffffffu, acc[i][d].y, o);
            }
}
}  // namespace

// KEYS = false: dq and the statistics.  KEYS = true: dk and dv.  grid (heads x tiles, 1, CTAs per tile)
// LIES: dout is read as it comes back from a projection, the heads of a token side by side, [B, L, H, DV], which saves a copy and
// its launch ahead (steps of B1 H8 L200 d_v 128 on the host 107 -> 105 us).  An instance of its own: with the distance of dout's
// rows as an argument the others were 1 % slower.
template <int DV, bool KEYS, bool LIES>
__global__ void __launch_bounds__(kBT, DV > 64 ? 1 : 2)
    backward_f32_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                        const float* __restrict__ g, float2* stats, float* __restrict__ dx, float* __restrict__ dv, int heads,
                        int L, int numerator_only, int dout_H) {
    using S = BwdSmem<DV, KEYS>;
    constexpr int NV = S::kCols / 64;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S& s = *reinterpret_cast<S*>(smem_raw);
    cg::cluster_group cluster = cg::this_cluster();
    const int nsplit = gridDim.z, rank = blockIdx.z, ntile = (L + kT - 1) / kT, turn = blockIdx.x / heads;
    const int own = KEYS ? turn : ntile - 1 - turn;                  // longest loops of all heads first
    const size_t head = blockIdx.x - turn * heads;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ro = lane & 1, co = lane >> 1;                         // pair tile: own rows row0 + {0..3, 8..11}, looped 4 co + j
    const int row0 = warp * 16 + ro * 4;
    const int dg = lane & 1, rg = (lane >> 1) & 3, ks = lane >> 3;   // narrow products
    const size_t hn = head * (size_t)L * kDFeat, hw = head * (size_t)L * DV;
    const float* own_n = (KEYS ? k : q) + hn;
    const size_t seq = LIES ? head / dout_H : 0, gw = LIES ? (seq * L * dout_H + head - seq * dout_H) * DV : hw;
    const size_t gp = LIES ? (size_t)dout_H * DV : DV, own_p = KEYS ? DV : gp, loop_p = KEYS ? gp : DV;
    const float* own_w = (KEYS ? v : g) + (KEYS ? hw : gw);
    const float* loop_n = (KEYS ? q : k) + hn;
    const float* loop_w = (KEYS ? g : v) + (KEYS ? gw : hw);
    const int n_own = min(kT, L - own * kT);

    load_tile<kDFeat>(s.an, nullptr, 0, false, own_n + (size_t)own * kT * kDFeat, n_own, warp, lane);
    load_tile<DV, LIES && !KEYS>(s.aw, nullptr, 0, false, own_w + (size_t)own * kT * own_p, n_own, warp, lane, own_p);
    float m[8];
    if (!KEYS) {
        // the centre m_i: two threads per row
        float x = 0.f;
        const int t = tid >> 1;
        if (t < n_own && !numerator_only) {
            const float4* gr = reinterpret_cast<const float4*>(g + gw + (size_t)(own * kT + t) * gp);
            const float4* vr = reinterpret_cast<const float4*>(v + hw + (size_t)(own * kT + t) * DV);
#pragma unroll 8
            for (int c = tid & 1; c < DV / 4; c += 2) {
                const float4 a = __ldg(gr + c), b = __ldg(vr + c);
                x = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, x))));
            }
        }
        x += __shfl_xor_sync(0xffffffffu, x, 1);
        if ((tid & 1) == 0) s.m[t] = x;
        __syncwarp();                                                // a warp's rows are its own
#pragma unroll
        for (int i = 0; i < 8; ++i) m[i] = s.m[row0 + (i >> 2) * 8 + (i & 3)];
    }

    float2 n1[4][4], n2[KEYS ? 1 : 4][4];            // X and Y, or dk
    float den[8], num[8];                            // row sums of w and w G.v (dq pass)
    float2 wide[KEYS ? 4 : 1][KEYS ? 4 * NV : 1];    // dv, rows in pairs
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int d = 0; d < 4; ++d) {
            n1[i][d] = make_float2(0.f, 0.f);
            if (!KEYS) n2[i][d] = make_float2(0.f, 0.f);
        }
#pragma unroll
    for (int i = 0; i < 8; ++i) den[i] = num[i] = 0.f;
    if (KEYS)
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < 4 * NV; ++c) wide[i][c] = make_float2(0.f, 0.f);

    float* p = s.p[warp];
    const int first = KEYS ? own : 0, last = KEYS ? ntile - 1 : own;
    for (int tile = first + rank; tile <= last; tile += nsplit) {
        const int n_loop = min(kT, L - tile * kT);
        __syncthreads();                             // the tile before is read
        load_tile<kDFeat>(s.bn, s.rn, kDFeat, true, loop_n + (size_t)tile * kT * kDFeat, n_loop, warp, lane);
        load_tile<DV, LIES && KEYS>(s.bw, KEYS ? s.rw : nullptr, S::kWide, false, loop_w + (size_t)tile * kT * loop_p, n_loop, warp, lane, loop_p);
        if (KEYS && tid < kT)
            s.st[tid] = tid < n_loop ? stats[head * (size_t)L + tile * kT + tid] : make_float2(0.f, 0.f);
        __syncthreads();

        float2 sc2[4][4], gv2[4][4];                 // rows in pairs
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) sc2[i][j] = gv2[i][j] = make_float2(0.f, 0.f);
        pair_product<kDFeat>(sc2, s.an + row0, s.bn + 4 * co);
        pair_product<DV>(gv2, s.aw + row0, s.bw + 4 * co);
        float sc[8][4], gv[8][4];
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                sc[i][j] = i & 1 ? sc2[i >> 1][j].y : sc2[i >> 1][j].x;
                gv[i][j] = i & 1 ? gv2[i >> 1][j].y : gv2[i >> 1][j].x;
            }

        const bool diag = tile == own;
        float2 st[4];
        if (KEYS)
#pragma unroll
            for (int j = 0; j < 4; ++j) st[j] = s.st[4 * co + j];
        // the first weight to the warp's shared memory; the second one takes the place of the scores.  MASKED: the own tile,
        // where pairs are left out by selection, not by a zero factor: a non-finite v or dout stays out of rows that do not
        // see it (selections in every tile: B2 H16 L1024 d_v64 272.6 -> 277 us)
        auto weigh = [&](auto masked_tag) {
            constexpr bool MASKED = decltype(masked_tag)::value;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float a[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int r = row0 + (i >> 2) * 8 + (i & 3), c = 4 * co + j;
                    const bool live = !MASKED || (KEYS ? r <= c : c <= r);
                    const float x = sc[i][j];
                    const float w = live ? fmaf(x, fmaf(x, 0.03125f, 0.25f), 1.0f) : 0.f;
                    const float w1 = fmaf(x, 0.0625f, 0.25f);
                    if (KEYS) {
                        a[i] = live ? fmaf(gv[i][j], st[j].x, st[j].y) * w1 : 0.f;
                        sc[i][j] = w * st[j].x;
                    } else {
                        den[i] += w;
                        if (live) num[i] = fmaf(w, gv[i][j], num[i]);
                        a[i] = live ? w1 * (gv[i][j] - m[i]) : 0.f;
                        sc[i][j] = live ? w1 : 0.f;
                    }
                }
                store_weight(p, a, j, co, ro);
            }
        };
        if (diag) weigh(std::true_type{});
        else weigh(std::false_type{});
        __syncwarp();
        narrow_product(n1, p, s.rn, ks, rg, dg);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float a[8] = {sc[0][j], sc[1][j], sc[2][j], sc[3][j], sc[4][j], sc[5][j], sc[6][j], sc[7][j]};
            store_weight(p, a, j, co, ro);
        }
        __syncwarp();
        if constexpr (!KEYS) {
            narrow_product(n2, p, s.rn, ks, rg, dg);
        } else {
            // dv rows row0 + ..., columns 64 c + 4 co + e
#pragma unroll 4
            for (int t = 0; t < kT; ++t) {
                const float* pr = p + place_of(t) * 16 + ro * 4;
                const float4 x0 = lds4(pr), x1 = lds4(pr + 8);
#pragma unroll
                for (int c = 0; c < NV; ++c) {
                    const float4 y = lds4(&s.rw[t * S::kWide + 64 * c + 4 * co]);
                    const float ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        fma_pair(wide[0][4 * c + e], x0.x, x0.y, ys[e]);
                        fma_pair(wide[1][4 * c + e], x0.z, x0.w, ys[e]);
                        fma_pair(wide[2][4 * c + e], x1.x, x1.y, ys[e]);
                        fma_pair(wide[3][4 * c + e], x1.z, x1.w, ys[e]);
                    }
                }
            }
        }
        __syncwarp();
    }

    // ---- sums to shared memory ([64][16] each, statistics, [64][DV]; s.m lies behind them), then out, each CTA of the
    // cluster its share of rows
    __syncthreads();
    float* o1 = reinterpret_cast<float*>(smem_raw);
    float* o2 = o1 + kT * kDFeat;
    float2* o3 = reinterpret_cast<float2*>(o2 + kT * kDFeat);
    float* ow = o2;                                  // keys pass: dv behind dk
    narrow_reduce(n1);
    if constexpr (!KEYS) narrow_reduce(n2);
    if (ks == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int at = (warp * 16 + rg * 4 + i) * kDFeat + dg * 8;
            *reinterpret_cast<float4*>(o1 + at) = make_float4(n1[i][0].x, n1[i][0].y, n1[i][1].x, n1[i][1].y);
            *reinterpret_cast<float4*>(o1 + at + 4) = make_float4(n1[i][2].x, n1[i][2].y, n1[i][3].x, n1[i][3].y);
            if constexpr (!KEYS) {
                *reinterpret_cast<float4*>(o2 + at) = make_float4(n2[i][0].x, n2[i][0].y, n2[i][1].x, n2[i][1].y);
                *reinterpret_cast<float4*>(o2 + at + 4) = make_float4(n2[i][2].x, n2[i][2].y, n2[i][3].x, n2[i][3].y);
            }
        }
    }
    if constexpr (!KEYS) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int o = 2; o < 32; o <<= 1) {
                den[i] += __shfl_xor_sync(0xffffffffu, den[i], o);
                num[i] += __shfl_xor_sync(0xffffffffu, num[i], o);
            }
        if (co == 0)
#pragma unroll
            for (int i = 0; i < 8; ++i) o3[row0 + (i >> 2) * 8 + (i & 3)] = make_float2(den[i], num[i]);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
            for (int c = 0; c < NV; ++c)
                if (64 * c + 4 * co < DV)
                    *reinterpret_cast<float4*>(ow + (row0 + (i >> 2) * 8 + (i & 3)) * DV + 64 * c + 4 * co) =
                        i & 1 ? make_float4(wide[i >> 1][4 * c].y, wide[i >> 1][4 * c + 1].y, wide[i >> 1][4 * c + 2].y, wide[i >> 1][4 * c + 3].y)
                              : make_float4(wide[i >> 1][4 * c].x, wide[i >> 1][4 * c + 1].x, wide[i >> 1][4 * c + 2].x, wide[i >> 1][4 * c + 3].x);
    }
    if (nsplit > 1) cluster.sync();
    else __syncthreads();
    auto sum4 = [&](float* p) {
        float4 x = lds4(p);
        if (nsplit > 1) {
            x = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int r = 0; r < nsplit; ++r) {
                const float4 y = *reinterpret_cast<const float4*>(cluster.map_shared_rank(p, r));
                x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
            }
        }
        return x;
    };
    const int share = kT / nsplit, r0 = rank * share;
    if constexpr (!KEYS) {
        const int r_end = min(r0 + share, n_own);
        for (int e = tid; e < share * 4; e += kBT) {
            const int r = r0 + (e >> 2), d = (e & 3) * 4;
            if (r >= r_end) continue;
            const float4 x = sum4(o1 + r * kDFeat + d), y = sum4(o2 + r * kDFeat + d);
            float dsum = 0.f, nsum = 0.f;
            for (int c = 0; c < nsplit; ++c) {
                const float2 t = nsplit > 1 ? *cluster.map_shared_rank(o3 + r, c) : o3[r];
                dsum += t.x;
                nsum += t.y;
            }
            const float inv = numerator_only ? 1.f : 1.f / (dsum + kEps);
            const float b = numerator_only ? 0.f : -nsum * inv * inv;
            const float c = numerator_only ? 0.f : fmaf(s.m[r], inv, b);
            *reinterpret_cast<float4*>(dx + hn + (size_t)(own * kT + r) * kDFeat + d) =
                make_float4(fmaf(x.x, inv, c * y.x), fmaf(x.y, inv, c * y.y), fmaf(x.z, inv, c * y.z), fmaf(x.w, inv, c * y.w));
            if (d == 0) stats[head * (size_t)L + own * kT + r] = make_float2(inv, b);
        }
    } else {
        const int r_end = min(r0 + share, n_own);
        for (int e = tid; e < share * 4; e += kBT) {
            const int r = r0 + (e >> 2), d = (e & 3) * 4;
            if (r < r_end)
                *reinterpret_cast<float4*>(dx + hn + (size_t)(own * kT + r) * kDFeat + d) = sum4(o1 + r * kDFeat + d);
        }
        for (int e = tid; e < share * (DV / 4); e += kBT) {
            const int r = r0 + e / (DV / 4), d = e % (DV / 4) * 4;
            if (r < r_end) *reinterpret_cast<float4*>(dv + hw + (size_t)(own * kT + r) * DV + d) = sum4(ow + r * DV + d);
        }
    }
    if (nsplit > 1) cluster.sync();                  // no CTA leaves while another reads its sums
}

namespace {
template <int DV, bool KEYS, bool LIES>
based_status launch_pass(const float* q, const float* k, const float* v, const float* g, float2* stats, float* dx, float* dv,
                         int BH, int L, int numerator_only, int dout_H, cudaStream_t stream) {
    const int smem = (int)sizeof(BwdSmem<DV, KEYS>);
    {
        static bool configured[64] = {};
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BASED_ERR_CUDA;
        std::lock_guard<std::mutex> lock(setup_mutex());
        if (!configured[dev]) {
            if (cudaFuncSetAttribute(backward_f32_kernel<DV, KEYS, LIES>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) !=
                cudaSuccess)
                return BASED_ERR_CUDA;
            configured[dev] = true;
        }
    }
    const int ntile = (L + kT - 1) / kT;
    // CTAs per own tile: as many as one wave of two per SM has room for, and two up to twice that, where one per tile leaves
    // a second wave of few (1 / 2 / 4 CTAs, us: 256 tiles of B1 H16 L1024 192 / 156 / 180, 224 of B2 H16 L390 87 / 83 / 103,
    // 512 of B4 H16 L512 151 / 176 / 232, 64 of B1 H8 L512 86 / 51 / 37)
    const long long tiles = (long long)BH * ntile;
    int nsplit = 1;
    while (nsplit < kMaxSplit && 2 * nsplit <= ntile && tiles * 2 * nsplit <= (nsplit == 1 ? 4 : 2) * kSMs) nsplit *= 2;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)BH * ntile, 1, nsplit);
    cfg.blockDim = dim3(kBT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = nsplit;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, backward_f32_kernel<DV, KEYS, LIES>, q, k, v, g, stats, dx, dv, BH, L, numerator_only, dout_H);
    note_launch();
    const based_status st = check_launch("backward_f32_kernel");
    return e == cudaSuccess ? st : BASED_ERR_CUDA;
}
template <int DV, bool LIES>
based_status launch_dv(const float* q, const float* k, const float* v, const float* g, float* dq, float* dk, float* dv,
                       float2* stats, int BH, int L, int numerator_only, int dout_H, cudaStream_t stream) {
    const based_status st = launch_pass<DV, false, LIES>(q, k, v, g, stats, dq, nullptr, BH, L, numerator_only, dout_H, stream);
    if (st != BASED_OK) return st;
    return launch_pass<DV, true, LIES>(q, k, v, g, stats, dk, dv, BH, L, numerator_only, dout_H, stream);
}
}  // namespace

based_status launch_prefill_backward_f32(const float* q, const float* k, const float* v, const float* g, int dout_H, float* dq,
                                         float* dk, float* dv, float* stats, int BH, int L, int d_v, int numerator_only,
                                         cudaStream_t stream) {
    auto launch = [&](auto lies) {
        constexpr bool LIES = decltype(lies)::value;
        float2* st = reinterpret_cast<float2*>(stats);
        if (d_v == 64) return launch_dv<64, LIES>(q, k, v, g, dq, dk, dv, st, BH, L, numerator_only, dout_H, stream);
        if (d_v == 112) return launch_dv<112, LIES>(q, k, v, g, dq, dk, dv, st, BH, L, numerator_only, dout_H, stream);
        return launch_dv<128, LIES>(q, k, v, g, dq, dk, dv, st, BH, L, numerator_only, dout_H, stream);
    };
    return dout_H ? launch(std::true_type{}) : launch(std::false_type{});
}

}  // namespace based
