// based_prefill for fp32 io (d' = 16): causal Taylor linear attention in chunked form with fp32 FMAs, the sequence of a
// head spread over the CTAs of one thread-block cluster.
//
// Tensor-core operand formats (bf16, tf32) cannot meet fp32's tolerance, so the contractions are register-tiled products
// on the fp32 pipe (two-wide fma.rn.f32x2), fed from shared memory.  One CTA holds 64 value columns of one sequence
// segment; the cluster's CTAs are the segments of a head in order (and, above 64 columns, its column groups):
//   1. every segment sums its own state  S_seg = sum_j psi(k_j) v_j^T  (153 features, one per unordered pair) and z_seg,
//      and leaves it in shared memory;
//   2. the cluster turns these sums, on top of the caller's state, into running sums in place: every CTA takes a share of
//      the elements through all segments' shared memory and writes that share of the final state (no scratch in global
//      memory, one launch);
//   3. chunks of 64 tokens: out = (psi(Q) S + P V) / (psi(Q) z + rowsum P), P = (1 + s/4 + s^2/32)[j <= i] with
//      s = q.k, then, unless it is the segment's last chunk, S += psi(K)^T V, z += sum psi(K).  A warp builds the feature
//      rows and weights of its own 8 query rows and is the only one that reads them.
// With one segment there is no step 1 and 2 and every chunk of step 3 updates the state.
// Bound: shared-memory passes and the fp32 pipe together (ncu, 296 heads x 512, d_v 64: 76 % of the shared-memory passes,
// 49 % of the FMA pipe's cycles; per chunk and SM 28 k cycles against 13 k of FMAs); at few heads the chain of chunks.
// Measured against one CTA per head that walked the tokens one by one: B1 H2 L256 d_v64 190 -> 22 us, B2 H16 L1024 d_v64
// 660 -> 92 us.
#include <cooperative_groups.h>

#include "common.cuh"
#include "f32_tiles.cuh"

namespace based {

namespace {
namespace cg = cooperative_groups;

constexpr int kTok = 64;           // tokens per chunk
constexpr int kNT = 256;
constexpr int kMaxSeg = 16;        // CTAs of the largest cluster

struct F32Smem {
    float psi[kFeatRows * kRowT];  // psi(K)^T [160][68], or psi(Q) [64][156] whose rows are replaced by P's [64][156]
    float st[64 * kFeat];          // state transposed: [64 columns][156 features]
    float z[kFeatRows];
    float vt[64 * kRowT];          // V^T of the chunk [64 columns][68]
    float xq[kTok * kRowX], xk[kTok * kRowX];
    FeatTab tab;
};
static_assert(sizeof(F32Smem) + 1024 <= (227 * 1024) / 2, "two CTAs per SM");
static_assert(kTok * kFeat <= kFeatRows * kRowT, "psi(Q) fits");

// The head's state in the caller's arrays, by symmetric feature f (order of based_decode_step_sym): the row itself, or the
// rows (m, n) and (n, m) of a full state.
struct AbiState {
    float* kv;                     // the head's first row, first column of this CTA
    float* z;
    int pitch;
    bool sym, keep;                // keep: a full state whose rows (m, n) and (n, m) differ keeps the difference
    __device__ __forceinline__ void rows(const FeatTab& tab, int f, int& a, int& b) const {
        a = b = f;
        if (sym || f <= kDFeat) return;
        const int m = tab.mn[f] & 255, n = tab.mn[f] >> 8;
        a = 1 + kDFeat + m * kDFeat + n;
        b = 1 + kDFeat + n * kDFeat + m;
    }
    static __device__ __forceinline__ float get(const float* p, size_t a, size_t b) {
        return a == b ? p[a] : (p[a] + p[b]) * kRsqrt2;
    }
    __device__ __forceinline__ void put(float* p, size_t a, size_t b, float x, bool pair) const {
        if (!pair) {
            p[a] = x;
            return;
        }
        const float half = keep ? 0.5f * (p[a] - p[b]) : 0.f;
        p[a] = fmaf(x, kRsqrt2, half);
        p[b] = fmaf(x, kRsqrt2, -half);
    }
    __device__ __forceinline__ float kv_get(const FeatTab& tab, int f, int c) const {
        int a, b;
        rows(tab, f, a, b);
        return get(kv + c, (size_t)a * pitch, (size_t)b * pitch);
    }
    __device__ __forceinline__ void kv_put(const FeatTab& tab, int f, int c, float x) const {
        int a, b;
        rows(tab, f, a, b);
        put(kv + c, (size_t)a * pitch, (size_t)b * pitch, x, a != b);
    }
    __device__ __forceinline__ float z_get(const FeatTab& tab, int f) const {
        int a, b;
        rows(tab, f, a, b);
        return get(z, a, b);
    }
    __device__ __forceinline__ void z_put(const FeatTab& tab, int f, float x) const {
        int a, b;
        rows(tab, f, a, b);
        put(z, a, b, x, a != b);
    }
};

// outputs of up to 8 NI tokens of a chunk; everything but the state, V^T and the k rows is the warp's own
template <int NI>
__device__ __forceinline__ void chunk_outputs(F32Smem& s, float* __restrict__ o, int d_v, int ncol, int nt, bool numerator_only,
                                              int warp, int lane) {
    psi_rows<NI>(s.psi, s.xq, s.tab, warp, lane);
    // weights of the rows warp + 8 i and the keys lane + 32 j
    float2 acc[NI][2];
    float p[NI][2], den[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
    rows_product<NI, kRowX, kRowX>(acc, s.xq, s.xk, kDFeat, warp, lane);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float x = acc[i][j].x + acc[i][j].y;
            p[i][j] = lane + 32 * j <= warp + 8 * i ? fmaf(x, fmaf(x, 0.03125f, 0.25f), 1.0f) : 0.f;
            acc[i][j] = make_float2(0.f, 0.f);
        }
        den[i] = p[i][0] + p[i][1];
    }
    __syncwarp();
    rows_product<NI, kFeat, kFeat>(acc, s.psi, s.st, kFeat, warp, lane);
    // cross-chunk denominator
#pragma unroll
    for (int u = 0; u < kTF; ++u) {
        const int f = lane + 32 * u;
        if (f < kFeat) {
            const float zf = s.z[f];
#pragma unroll
            for (int i = 0; i < NI; ++i) den[i] = fmaf(s.psi[(warp + 8 * i) * kFeat + f], zf, den[i]);
        }
    }
    __syncwarp();                                    // psi(Q) is read: P takes its place
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        den[i] = warp_sum(den[i]);
        s.psi[(warp + 8 * i) * kFeat + lane] = p[i][0];
        s.psi[(warp + 8 * i) * kFeat + lane + 32] = p[i][1];
    }
    __syncwarp();
    rows_product<NI, kFeat, kRowT>(acc, s.psi, s.vt, (nt + 3) & ~3, warp, lane);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int t = warp + 8 * i;
        if (t >= nt) continue;
        const float d = numerator_only ? 1.f : den[i] + kEps;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int c = lane + 32 * j;
            if (c < ncol) o[(size_t)t * d_v + c] = (acc[i][j].x + acc[i][j].y) / d;
        }
    }
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
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int t_begin = min(rank * seg, L), t_end = min(t_begin + seg, L);
    const bool cont = (flags & BASED_STATE_CONTINUE) != 0, numerator_only = (flags & BASED_NUMERATOR_ONLY) != 0;
    AbiState abi;
    abi.sym = (flags & BASED_STATE_SYM) != 0;
    abi.keep = cont && !abi.sym;
    abi.pitch = d_v;
    abi.kv = kv + head * (size_t)(abi.sym ? kDSym : kD) * d_v + col0;
    abi.z = z + head * (size_t)(abi.sym ? kDSym : kD);

    const float* qh = q + head * (size_t)L * kDFeat;
    const float* kh = k + head * (size_t)L * kDFeat;
    const float* vh = v + head * (size_t)L * d_v + col0;
    float* oh = out + head * (size_t)L * d_v + col0;

    fill_feat_tab(s.tab, tid);
    __syncthreads();

    // a chunk's contribution to the state tile of a thread: features lane + 32 i, columns 8 warp + j
    auto chunk_state = [&](float2 (&acc)[kTF][8], int nt) {
        psi_transposed(s.psi, s.xk, s.tab, nt, tid);
        __syncthreads();
        state_update(acc, s.psi, s.vt, nt, warp, lane);
    };
    float zsum = 0.f;                                // thread f < 160: z of feature f
    if (nseg > 1) {
        // ---- step 1: this segment's own state (the last one's is needed for the final state only)
        float2 acc[kTF][8];
#pragma unroll
        for (int i = 0; i < kTF; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = make_float2(0.f, 0.f);
        const float zc = cont && rank == 0 && tid < kDSym ? abi.z_get(s.tab, tid) : 0.f;
        if (rank < nseg - 1 || kv != nullptr) {
            for (int t0 = t_begin; t0 < t_end; t0 += kTok) {
                const int nt = min(kTok, t_end - t0);
                load_x(s.xk, kh + (size_t)t0 * kDFeat, nt, tid);
                load_vt(s.vt, vh + (size_t)t0 * d_v, d_v, ncol, nt, tid);
                __syncthreads();
                chunk_state(acc, nt);
                if (tid < kFeatRows) zsum += row_sum(s.psi, tid, nt);
                __syncthreads();
            }
        }
#pragma unroll
        for (int i = 0; i < kTF; ++i) {
            const int f = lane + 32 * i;
            if (f < kFeat)
#pragma unroll
                for (int j = 0; j < 8; ++j) s.st[(warp * 8 + j) * kFeat + f] = acc[i][j].x + acc[i][j].y;
        }
        if (tid < kFeatRows) s.z[tid] = zsum;
        cluster.sync();

        // ---- step 2: running sums over the segments, four features of a column per thread; consecutive lanes take
        // consecutive columns, so the caller's state is read and written in whole rows
        for (int e = rank * kNT + tid; e < 64 * (kFeat / 4); e += nseg * kNT) {
            const int c = e & 63, f = (e >> 6) * 4;
            float4* mine = reinterpret_cast<float4*>(&s.st[c * kFeat + f]);
            float4 x[kMaxSeg];
#pragma unroll
            for (int r = 0; r < kMaxSeg; ++r)
                if (r < nseg) x[r] = *cluster.map_shared_rank(mine, cluster_row + r);
            float run[4] = {0.f, 0.f, 0.f, 0.f};
            if (cont && c < ncol)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (f + u < kDSym) run[u] = abi.kv_get(s.tab, f + u, c);
#pragma unroll
            for (int r = 0; r < kMaxSeg; ++r)
                if (r < nseg) {
                    *cluster.map_shared_rank(mine, cluster_row + r) = make_float4(run[0], run[1], run[2], run[3]);
                    run[0] += x[r].x; run[1] += x[r].y; run[2] += x[r].z; run[3] += x[r].w;
                }
            if (kv != nullptr && c < ncol)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (f + u < kDSym) abi.kv_put(s.tab, f + u, c, run[u]);
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
        cluster.sync();
    } else {
        for (int e = tid; e < 64 * kFeat; e += kNT) {
            const int c = e & 63, f = e >> 6;
            s.st[c * kFeat + f] = cont && f < kDSym && c < ncol ? abi.kv_get(s.tab, f, c) : 0.f;
        }
        if (tid < kFeatRows) s.z[tid] = cont && tid < kDSym ? abi.z_get(s.tab, tid) : 0.f;
        // column group 0 writes the K-state that the other one reads
        if (cont && gridDim.z > 1) cluster.sync();
    }

    // ---- step 3: outputs, chunk by chunk
    for (int t0 = t_begin; t0 < t_end; t0 += kTok) {
        const int nt = min(kTok, t_end - t0);
        load_x(s.xq, qh + (size_t)t0 * kDFeat, nt, tid);
        load_x(s.xk, kh + (size_t)t0 * kDFeat, nt, tid);
        load_vt(s.vt, vh + (size_t)t0 * d_v, d_v, ncol, nt, tid);
        __syncthreads();
        float* o = oh + (size_t)t0 * d_v;
        if (nt > 32) chunk_outputs<8>(s, o, d_v, ncol, nt, numerator_only, warp, lane);
        else if (nt > 16) chunk_outputs<4>(s, o, d_v, ncol, nt, numerator_only, warp, lane);
        else chunk_outputs<2>(s, o, d_v, ncol, nt, numerator_only, warp, lane);
        if (t0 + kTok >= t_end && (nseg > 1 || kv == nullptr)) break;   // nobody reads the state after this chunk
        __syncthreads();                             // P and the state are read
        float2 acc[kTF][8];
#pragma unroll
        for (int i = 0; i < kTF; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[i][j] = make_float2(0.f, 0.f);
        chunk_state(acc, nt);
#pragma unroll
        for (int i = 0; i < kTF; ++i) {
            const int f = lane + 32 * i;
            if (f < kFeat)
#pragma unroll
                for (int j = 0; j < 8; ++j) s.st[(warp * 8 + j) * kFeat + f] += acc[i][j].x + acc[i][j].y;
        }
        if (tid < kFeatRows) s.z[tid] += row_sum(s.psi, tid, nt);
        __syncthreads();
    }

    if (nseg == 1 && kv != nullptr) {
        for (int e = tid; e < 64 * kDSym; e += kNT) {
            const int c = e & 63, f = e >> 6;
            if (c < ncol) abi.kv_put(s.tab, f, c, s.st[c * kFeat + f]);
        }
        if (blockIdx.z == 0 && tid < kDSym) abi.z_put(s.tab, tid, s.z[tid]);
    }
}

namespace {
// whole groups of 16 tokens, so that every segment but the last ends on a tile edge of the products
int f32_segment_tokens(int L, int nseg) { return ((L + nseg - 1) / nseg + 15) / 16 * 16; }
// Segments per head (the cluster holds all segments of both column groups, at most 16 CTAs), by a time model fitted on
// B200, in us: outputs of a full chunk 10.5 (a chunk of up to 32 / 16 tokens 0.5 / 0.3 of that), a state update 5.5, two
// CTAs on an SM 1.9 times one, 5 for launch and ramps, 4 + 0.3 n for the running sums of n segments, all of it once per
// wave.  Clusters of 8 and 16 CTAs leave SMs of a GPC unused: about 104 and 96 fit one per SM.  More segments shorten the
// chain of chunks but every chunk then updates a state twice (its segment's own sums, then the running state): B1 H2 L256
// d_v64 70 / 46 / 26 / 23 / 22 us with 1 / 2 / 4 / 8 / 16 segments, B2 H16 L1024 d_v64 257 / 177 / 92 / 93 / 126, B8 H16
// L512 d_v64 133 / 153 / 150 / 184 / 343, B1 H16 L700 d_v64 179 / 126 / 68 / 71 / 75.  The same whether the state is asked
// for or not: so are the outputs.
int f32_segments(int BH, int L, int nz) {
    int best = 1;
    double best_t = 1e30;
    for (int n = 1; n * nz <= kMaxSeg; n *= 2) {
        const int seg = f32_segment_tokens(L, n), rest = seg % kTok, chunks = (seg + kTok - 1) / kTok;
        const double outs = seg / kTok + (rest == 0 ? 0.0 : rest <= 16 ? 0.3 : rest <= 32 ? 0.5 : 1.0);
        const double ups = n > 1 ? 2 * chunks - 1 : chunks;
        const long long ctas = (long long)BH * nz * n, fit = n * nz <= 4 ? 148 : n * nz == 8 ? 104 : 96;
        const double waves = (double)((ctas + 2 * fit - 1) / (2 * fit));
        const double t = waves * ((ctas <= fit ? 1.0 : 1.9) * (outs * 10.5 + ups * 5.5) + 5.0 + (n > 1 ? 4.0 + 0.3 * n : 0.0));
        if (t < best_t) { best_t = t; best = n; }
    }
    return best;
}
}  // namespace

based_status launch_prefill_f32(const void* q, const void* k, const void* v, void* out, float* kv, float* z, int BH,
                                int L, int d_v, int flags, cudaStream_t stream) {
    const int nz = d_v > 64 ? 2 : 1, ncol = d_v / nz;        // 64 or (d_v 112) 56 columns per CTA
    const int nseg = f32_segments(BH, L, nz), seg = f32_segment_tokens(L, nseg);
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
