// based_generation_step: one generated token through both mixers of a Based layer pair in ONE launch.
//
// The linear-attention decode step (Sec. 4.1 recurrences, Algorithm 2) streams each head's fp32 state once;
// the sliding-window decode step (Algorithm 3) reads a small rolling cache.  The paper runs next-token
// prediction under CUDA graphs (Sec. 6, "Efficiency Benchmarks") because at these sizes launch and fill
// latencies are a visible share of a step.  As two kernels, even as two branches of one graph, the short
// window step runs after (or before) the long state stream: the state kernel's CTAs fill every SM's
// register file, so the other kernel's CTAs wait for a wave to drain.  Here both kinds of CTA are one
// grid, dealt out in turn (one window CTA, holding two heads, per two state CTAs), so the window heads'
// bulk copies and their fill and drain latency ride in the shadow of the state stream and the step costs
// one launch.
//
// CTA roles by block index (256 threads each):
//   window role: two groups of 128 threads, one head each, the code of swa_decode_kernel with a named
//                barrier per group (swa_decode.cuh);
//   state role:  the code of decode_step_kernel (decode.cuh), with few heads shared by the CTAs of a cluster as there.
// A dependent launch: its CTAs come in while the grid ahead drains and wait for it before they read anything (steps back to back,
// 153 rows, d_v 128, 128 / 256 / 512 / 1024 state heads: 8.7 / 12.3 / 18.5 / 32.7 us plain, 8.1 / 10.1 / 16.7 / 30.4).
#include "decode.cuh"
#include "swa_decode.cuh"

namespace based {

namespace {
using namespace swa_dec;

struct GenArgs {
    // linear attention
    const void *q, *k, *v;
    float *kv, *z;
    void* out;
    int n_lin;            // heads
    int numerator_only;
    // sliding window
    const void *qw, *kw, *vw;
    void *kc, *vc, *outw;
    int n_swa;            // heads
    int window;
    int* pos_state;       // {position, ticket}
    float scale;
    unsigned int* err;
    int n_pairs;          // dealing of the roles: leading triples (window CTA, state CTA, state CTA)
    int swa_group_bytes;  // shared memory of one 128-thread window group
    void* keep[6];        // null, or where the step leaves a copy of q, k, v, qw, kw, vw
};

// head's W values of an input to the place where a copy is kept (threads of one warp)
template <typename T, int W>
__device__ __forceinline__ void keep_row(void* to, const void* from, size_t head, int lane) {
    for (int i = lane; i < W; i += 32) static_cast<T*>(to)[head * W + i] = static_cast<const T*>(from)[head * W + i];
}

template <int DV, typename T, bool STREAM, bool SYM, int NPW, int PARTS, int UN, int CTAS>
__global__ void __launch_bounds__(256, CTAS) generation_step_kernel(const GenArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    enter_dependent();
    // block index -> role: the first 3 * n_pairs blocks come in triples (window, state, state); then
    // whatever window CTAs are left, then the remaining state CTAs.  With PARTS > 1 a block of this numbering is a
    // cluster: the parts of one state head, or that many window CTAs.
    const int i = blockIdx.x / PARTS, part = blockIdx.x % PARTS, n_swa_ctas = ((a.n_swa + 1) / 2 + PARTS - 1) / PARTS;
    int swa_cta = -1, lin_head = -1;
    if (i < 3 * a.n_pairs) {
        const int g = i / 3, r = i - 3 * g;
        if (r == 0) swa_cta = g;
        else lin_head = 2 * g + r - 1;
    } else {
        const int j = i - 3 * a.n_pairs;
        if (j < n_swa_ctas - a.n_pairs) swa_cta = a.n_pairs + j;
        else lin_head = 2 * a.n_pairs + j - (n_swa_ctas - a.n_pairs);
    }
    if (swa_cta >= 0) {
        const int half = threadIdx.x >> 7;
        const int head = 2 * (swa_cta * PARTS + part) + half;
        if (head < a.n_swa) {
            const T* qw = static_cast<const T*>(a.qw);
            const T* kw = static_cast<const T*>(a.kw);
            const T* vw = static_cast<const T*>(a.vw);
            T* kc = static_cast<T*>(a.kc);
            T* vc = static_cast<T*>(a.vc);
            T* ow = static_cast<T*>(a.outw);
            // one named barrier per group (a compile-time id keeps the CTA's barrier count at three)
            if (half == 0)
                swa_decode_body<T, NPW, 1>(qw, kw, vw, kc, vc, ow, a.window, 0, a.pos_state, a.pos_state, a.scale, a.err,
                                           (size_t)head, threadIdx.x & 127, a.n_swa, smem);
            else
                swa_decode_body<T, NPW, 2>(qw, kw, vw, kc, vc, ow, a.window, 0, a.pos_state, a.pos_state, a.scale, a.err,
                                           (size_t)head, threadIdx.x & 127, a.n_swa, smem + a.swa_group_bytes);
            const int warp = (threadIdx.x & 127) >> 5, lane = threadIdx.x & 31;
            if (a.keep[3] != nullptr && warp < 3) {
                if (warp == 0) keep_row<T, kHD>(a.keep[3], a.qw, head, lane);
                else if (warp == 1) keep_row<T, kHD>(a.keep[4], a.kw, head, lane);
                else keep_row<T, kHD>(a.keep[5], a.vw, head, lane);
            }
        }
    } else {
        decode_step_body<DV, T, SYM, PARTS, UN, STREAM>(static_cast<const T*>(a.q), static_cast<const T*>(a.k),
                                                    static_cast<const T*>(a.v), a.kv, a.z, static_cast<T*>(a.out),
                                                    a.numerator_only, (size_t)lin_head, part);
        if (a.keep[0] != nullptr && part == 0) {
            const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
            if (warp == 0) keep_row<T, kDFeat>(a.keep[0], a.q, lin_head, lane);
            else if (warp == 1) keep_row<T, kDFeat>(a.keep[1], a.k, lin_head, lane);
            else if (warp == 2) keep_row<T, DV>(a.keep[2], a.v, lin_head, lane);
        }
    }
}

// State rows in flight per thread and CTAs per SM: 18 and 2, but 6 and 4 for narrow states that stay in L2 (batch 64 x 16
// heads, 153 rows, d_v 64: 12.2 against 13.5 us; d_v 128: 25.8 deep, 30.9 wide; batch 128: 53.8 deep, 67.6 wide, 57.6 before both).
template <int DV, bool STREAM> struct Depth {
    static constexpr bool kWide = DV == 64 && !STREAM;
    static constexpr int kRows = kWide ? 6 : 18, kCtas = kWide ? 4 : 2;
    // percent of an SM's 256 KB for shared memory, the rest is L1 for the loads in flight (batch 128, d_v 128, 153 rows:
    // 100 / 80 / 60 / 50 / 40 % 68.8 / 55.2 / 54.1 / 53.9 / 57.9 us; batch 64, d_v 64, 273 rows: 25.3 / 21.3 / 22.6 / 22.6 / 27.1)
    static constexpr int kShared = kWide ? 80 : 50;
};

template <int DV, typename T, bool STREAM, bool SYM, int NPW, int PARTS>
based_status launch_k(const GenArgs& args, size_t smem, cudaStream_t stream) {
    auto kern = generation_step_kernel<DV, T, STREAM, SYM, NPW, PARTS, (PARTS > 1 ? 9 : Depth<DV, STREAM>::kRows), Depth<DV, STREAM>::kCtas>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return BASED_ERR_CUDA;
    static std::atomic<bool> split[64];
    if (prefer_l1(kern, Depth<DV, STREAM>::kShared, split) != cudaSuccess) return BASED_ERR_CUDA;
    GenArgs a = args;
    const int n_swa_ctas = ((a.n_swa + 1) / 2 + PARTS - 1) / PARTS;
    a.n_pairs = n_swa_ctas < a.n_lin / 2 ? n_swa_ctas : a.n_lin / 2;
    const cudaError_t e = launch_ex(kern, dim3((a.n_lin + n_swa_ctas) * PARTS), dim3(256), smem, PARTS, true, stream, a);
    const based_status st = check_launch("generation_step_kernel");
    return e == cudaSuccess ? st : BASED_ERR_CUDA;
}

template <int DV, typename T, bool STREAM, bool SYM, int NPW>
based_status launch_p(const GenArgs& a, size_t smem, cudaStream_t stream) {
    if constexpr (!STREAM) {
        const int parts = decode_parts<DV, SYM>(a.n_lin);
        if (parts == 8) return launch_k<DV, T, STREAM, SYM, NPW, 8>(a, smem, stream);
        if (parts == 4) return launch_k<DV, T, STREAM, SYM, NPW, 4>(a, smem, stream);
        if (parts == 2) return launch_k<DV, T, STREAM, SYM, NPW, 2>(a, smem, stream);
    }
    return launch_k<DV, T, STREAM, SYM, NPW, 1>(a, smem, stream);
}
template <int DV, typename T, bool STREAM, bool SYM>
based_status launch_w(const GenArgs& a, size_t smem, cudaStream_t stream) {
    return a.window <= 64 ? launch_p<DV, T, STREAM, SYM, 4>(a, smem, stream) : launch_p<DV, T, STREAM, SYM, 8>(a, smem, stream);
}
template <int DV, typename T>
based_status launch_s(const GenArgs& a, size_t smem, bool sym, bool streaming, cudaStream_t stream) {
    if (sym) return streaming ? launch_w<DV, T, true, true>(a, smem, stream) : launch_w<DV, T, false, true>(a, smem, stream);
    return streaming ? launch_w<DV, T, true, false>(a, smem, stream) : launch_w<DV, T, false, false>(a, smem, stream);
}
template <typename T>
based_status launch_d(const GenArgs& a, int d_v, bool sym, cudaStream_t stream) {
    const size_t group = (swa_decode_smem_bytes<T>(a.window) + 127) & ~(size_t)127;
    GenArgs b = a;
    b.swa_group_bytes = (int)group;
    const size_t smem = 2 * group;
    const bool streaming = decode_streams(a.n_lin, d_v, sym);
    if (d_v == 64) return launch_s<64, T>(b, smem, sym, streaming, stream);
    if (d_v == 112) return launch_s<112, T>(b, smem, sym, streaming, stream);
    return launch_s<128, T>(b, smem, sym, streaming, stream);
}
}  // namespace

namespace {
template <int DV, typename T, bool STREAM, bool SYM, int NPW, int PARTS>
bool load_parts() {
    auto kern = generation_step_kernel<DV, T, STREAM, SYM, NPW, PARTS, (PARTS > 1 ? 9 : Depth<DV, STREAM>::kRows), Depth<DV, STREAM>::kCtas>;
    cudaFuncAttributes attr;
    // the largest request a launch of this variant can make: two groups at the widest window it serves
    const size_t group = (swa_decode_smem_bytes<T>(NPW == 4 ? 64 : 128) + 127) & ~(size_t)127;
    return cudaFuncGetAttributes(&attr, kern) == cudaSuccess &&
           cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(2 * group)) == cudaSuccess;
}
template <int DV, typename T, bool STREAM, bool SYM, int NPW>
bool load_one() {
    if (!load_parts<DV, T, STREAM, SYM, NPW, 1>()) return false;
    if constexpr (!STREAM) return load_parts<DV, T, STREAM, SYM, NPW, 2>() && load_parts<DV, T, STREAM, SYM, NPW, 4>() && load_parts<DV, T, STREAM, SYM, NPW, 8>();
    return true;
}
template <int DV, typename T>
bool load_dv() {
    return load_one<DV, T, false, false, 4>() && load_one<DV, T, false, false, 8>() && load_one<DV, T, true, false, 4>() &&
           load_one<DV, T, true, false, 8>() && load_one<DV, T, false, true, 4>() && load_one<DV, T, false, true, 8>() &&
           load_one<DV, T, true, true, 4>() && load_one<DV, T, true, true, 8>();
}
}  // namespace

// Loads every variant into the current context and sets its shared-memory limit, so that a first use
// inside a stream capture does neither.
based_status preload_generation_step() {
    const bool ok = load_dv<64, float>() && load_dv<64, __nv_bfloat16>() && load_dv<112, float>() &&
                    load_dv<112, __nv_bfloat16>() && load_dv<128, float>() && load_dv<128, __nv_bfloat16>();
    return ok ? BASED_OK : BASED_ERR_CUDA;
}

namespace {
struct GenCall {
    GenArgs a;
    int d_v;
    bool sym;
    based_dtype io;
};
}  // namespace

size_t generation_step_args_bytes() { return sizeof(GenCall); }

based_status make_generation_args(void* args, const void* q, const void* k, const void* v, float* kv, float* z, void* out,
                                  int n_lin, int d_v, bool sym, bool numerator_only, const void* qw, const void* kw, const void* vw,
                                  void* kc, void* vc, void* outw, int n_swa, int window, int* pos_state, float scale,
                                  based_dtype io) {
    GenCall& c = *static_cast<GenCall*>(args);
    GenArgs& a = c.a;
    a = GenArgs{};
    a.q = q; a.k = k; a.v = v; a.kv = kv; a.z = z; a.out = out; a.n_lin = n_lin; a.numerator_only = numerator_only ? 1 : 0;
    a.qw = qw; a.kw = kw; a.vw = vw; a.kc = kc; a.vc = vc; a.outw = outw; a.n_swa = n_swa; a.window = window;
    a.pos_state = pos_state; a.scale = scale;
    c.d_v = d_v; c.sym = sym; c.io = io;
    return error_word_ptr(&a.err) == BASED_OK ? BASED_OK : BASED_ERR_CUDA;
}

based_status launch_generation_args(const void* args, cudaStream_t stream) {
    const GenCall& c = *static_cast<const GenCall*>(args);
    return c.io == BASED_F32 ? launch_d<float>(c.a, c.d_v, c.sym, stream) : launch_d<__nv_bfloat16>(c.a, c.d_v, c.sym, stream);
}

based_status launch_generation_step(const void* q, const void* k, const void* v, float* kv, float* z, void* out,
                                    int n_lin, int d_v, bool sym, bool numerator_only, const void* qw, const void* kw,
                                    const void* vw, void* kc, void* vc, void* outw, int n_swa, int window,
                                    int* pos_state, float scale, based_dtype io, cudaStream_t stream) {
    GenCall c;
    const based_status st = make_generation_args(&c, q, k, v, kv, z, out, n_lin, d_v, sym, numerator_only, qw, kw, vw, kc, vc, outw,
                                                 n_swa, window, pos_state, scale, io);
    if (st != BASED_OK) return st;
    note_launch();
    return launch_generation_args(&c, stream);
}

void generation_step_inputs(void* args, const void* const* in, void* const* buffers) {
    GenArgs& a = static_cast<GenCall*>(args)->a;
    const void** const to[6] = {&a.q, &a.k, &a.v, &a.qw, &a.kw, &a.vw};
    for (int i = 0; i < 6; ++i) {
        *to[i] = in[i] ? in[i] : buffers[i];
        a.keep[i] = in[i] ? buffers[i] : nullptr;
    }
}

}  // namespace based
