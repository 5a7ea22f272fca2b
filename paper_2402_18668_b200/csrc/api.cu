// C ABI of libbased: argument validation and dispatch.  See include/based.h for the
// contract of every entry point.
#include <atomic>
#include <mutex>
#include <cstdio>
#include <new>
#include <vector>

#include "common.cuh"

namespace based {

__device__ unsigned int g_error_word = 0;

based_status error_word_ptr(unsigned int** ptr) {
    // the symbol has one instance per device: resolve it once per device, with that device current
    static std::atomic<unsigned int*> cache[64];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return BASED_ERR_CUDA;
    unsigned int* p = cache[dev].load(std::memory_order_acquire);
    if (p == nullptr) {
        void* q = nullptr;
        if (cudaGetSymbolAddress(&q, g_error_word) != cudaSuccess) return BASED_ERR_CUDA;
        p = static_cast<unsigned int*>(q);
        cache[dev].store(p, std::memory_order_release);
    }
    *ptr = p;
    return BASED_OK;
}

std::mutex& setup_mutex() {
    static std::mutex mu;
    return mu;
}

static std::atomic<unsigned long long> g_launches{0};

void note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }

based_status check_launch(const char* what) {
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        std::fprintf(stderr, "libbased: launch of %s failed: %s\n", what, cudaGetErrorString(e));
        return BASED_ERR_CUDA;
    }
    return BASED_OK;
}

static inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
// value head dimensions: 64 (360M-scale heads), 128, and 112 (the 1.3B configuration's 1792 / 16)
static inline bool dv_ok(int d_v) { return d_v == 64 || d_v == 112 || d_v == 128; }
// feature dimensions of the paper's ablation other than 16: served by the fp32 definition-form kernels
static inline bool df_generic(int d_feat) { return d_feat == 8 || d_feat == 24 || d_feat == 32; }

}  // namespace based

using namespace based;

// Several kernels index heads by the y dimension of the grid (at most 65535).  Larger batches are cut into
// slabs of heads here: every tensor is [B*H, ...] with the heads outermost, so a slab is a contiguous piece,
// and the slabs run one after another on the caller's stream (sharing the caller's workspace, which is sized
// for the largest slab).
constexpr long long kHeadSlab = 65532;      // a multiple of 4: a slab's K-state (an odd number of floats per head) stays 16-byte aligned
static inline const void* off(const void* p, size_t bytes) { return p ? static_cast<const char*>(p) + bytes : nullptr; }
static inline void* off(void* p, size_t bytes) { return p ? static_cast<char*>(p) + bytes : nullptr; }
static inline float* off(float* p, size_t floats) { return p ? p + floats : nullptr; }
static inline size_t esize(based_dtype io) { return io == BASED_BF16 ? 2 : 4; }

extern "C" {

int based_version(void) { return 1; }

unsigned long long based_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char* based_status_string(based_status s) {
    switch (s) {
        case BASED_OK: return "ok";
        case BASED_ERR_INVALID_ARG: return "invalid argument";
        case BASED_ERR_UNSUPPORTED: return "unsupported shape or dtype";
        case BASED_ERR_ALIGNMENT: return "pointer not 16-byte aligned";
        case BASED_ERR_CUDA: return "CUDA error";
        case BASED_ERR_DEVICE_TIMEOUT: return "bounded device-side wait timed out";
        case BASED_ERR_WORKSPACE: return "workspace missing or too small";
    }
    return "unknown status";
}

size_t based_prefill_workspace_bytes(int B, int H, int L, int d_feat, int d_v, based_dtype io) {
    if (B <= 0 || H <= 0 || L <= 0 || d_feat != kDFeat || !dv_ok(d_v)) return 0;
    if (io != BASED_BF16) return 0;            // the fp32 path keeps its states on chip
    const long long BH = (long long)B * H;
    if (BH > kHeadSlab) {
        const size_t a = prefill_tc_workspace_bytes((int)kHeadSlab, L, d_v);
        const size_t b = BH % kHeadSlab ? prefill_tc_workspace_bytes((int)(BH % kHeadSlab), L, d_v) : 0;
        return a > b ? a : b;
    }
    return prefill_tc_workspace_bytes(B * H, L, d_v);
}

size_t based_f32_parts_bytes(int B, int H, int L, int d_feat, int d_v, int backward) {
    if (B <= 0 || H <= 0 || L <= 0 || d_feat != kDFeat || !dv_ok(d_v)) return 0;
    const int heads = (long long)B * H > kHeadSlab ? (int)kHeadSlab : B * H;       // the largest slab of heads
    return quadratic_f32_workspace_bytes(heads, L, d_v, backward != 0);
}

static based_status prefill_impl(const void* q, const void* k, const void* v, void* out, float* kv_state, float* z_state,
                                 int B, int H, int L, int d_feat, int d_v, based_dtype io, int flags, void* workspace,
                                 size_t workspace_bytes, void* cuda_stream, bool fit) {
    if (!q || !k || !v || !out || B <= 0 || H <= 0 || L <= 0) return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (flags & ~(BASED_STATE_CONTINUE | BASED_STATE_SYM | BASED_NUMERATOR_ONLY)) return BASED_ERR_INVALID_ARG;
    if ((kv_state == nullptr) != (z_state == nullptr)) return BASED_ERR_INVALID_ARG;
    if ((flags & BASED_STATE_CONTINUE) && !kv_state) return BASED_ERR_INVALID_ARG;
    if (out == q || out == k || out == v) return BASED_ERR_INVALID_ARG;
    if ((d_feat != kDFeat && !df_generic(d_feat)) || !dv_ok(d_v)) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(kv_state) ||
        !aligned16(z_state) || !aligned16(workspace))
        return BASED_ERR_ALIGNMENT;
    if ((long long)B * H > kHeadSlab) {
        const size_t es = esize(io), rows = (flags & BASED_STATE_SYM) ? kDSym : 1 + d_feat + d_feat * d_feat;
        for (long long h0 = 0; h0 < (long long)B * H; h0 += kHeadSlab) {
            const int n = (int)((long long)B * H - h0 < kHeadSlab ? (long long)B * H - h0 : kHeadSlab);
            const based_status st = prefill_impl(
                off(q, (size_t)h0 * L * d_feat * es), off(k, (size_t)h0 * L * d_feat * es), off(v, (size_t)h0 * L * d_v * es),
                off(out, (size_t)h0 * L * d_v * es), off(kv_state, (size_t)h0 * rows * d_v), off(z_state, (size_t)h0 * rows),
                1, n, L, d_feat, d_v, io, flags, workspace, workspace_bytes, cuda_stream, fit);
            if (st != BASED_OK) return st;
        }
        return BASED_OK;
    }
    if (d_feat != kDFeat) {
        if (flags & BASED_STATE_SYM) return BASED_ERR_UNSUPPORTED;
        // bf16 io from the empty state: outputs (definition form) and state on the tensor cores, side by side
        if (io == BASED_BF16 && !(flags & BASED_STATE_CONTINUE)) {
            cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
            if (kv_state) {
                const based_status st = launch_state_generic_tc(k, v, kv_state, z_state, B * H, L, d_feat, d_v, 0, stream);
                if (st != BASED_OK) return st;
            }
            return launch_quadratic_forward_tc(q, k, v, out, B * H, L, d_feat, d_v, (flags & BASED_NUMERATOR_ONLY) ? 1 : 0,
                                               kv_state != nullptr, stream);
        }
        return launch_prefill_generic(q, k, v, out, kv_state, z_state, B * H, L, d_feat, d_v, io, flags,
                                      static_cast<cudaStream_t>(cuda_stream));
    }
    const size_t need = based_prefill_workspace_bytes(B, H, L, d_feat, d_v, io);
    if (!fit && need > 0 && (!workspace || workspace_bytes < need)) {
        // a few words for continued calls alone: others need none, and a continued call without them takes a plan without them
        if (need > BASED_WORDS_BYTES) return BASED_ERR_WORKSPACE;
        fit = true;
        if (!workspace) workspace_bytes = 0;
    }
    // One chunk and no state to write: the chunk's pairs are all there is, and the definition form's kernels, the same sums of the same
    // bf16 weights in the same order (the outputs are the bits that a call with a state gives), have less to set up (us, chunked / this: d_v 64, 16 heads L64 4.8 / 3.4, L128 5.7 / 3.8, 200 heads L64 10.6 / 4.0;
    // d_v 128, 16 heads L64 5.9 / 3.8, 400 heads L128 23 / 9).  Longer calls would be faster so up to L 1500 with 16 heads (L1024 10.2 /
    // 7.2), but the chunked form holds what is before the chunk more precisely (2.25e-3 against 2.29e-3 of 64-bit results).
    if (io == BASED_BF16 && !kv_state && L <= 128)
        return launch_quadratic_forward_tc(q, k, v, out, B * H, L, d_feat, d_v, (flags & BASED_NUMERATOR_ONLY) ? 1 : 0, false,
                                           static_cast<cudaStream_t>(cuda_stream));
    if (io == BASED_BF16)
        return launch_prefill_tc(q, k, v, out, kv_state, z_state, B * H, L, d_v, flags, workspace,
                                 static_cast<cudaStream_t>(cuda_stream), fit ? workspace_bytes : ~(size_t)0);
    return launch_prefill_f32(q, k, v, out, kv_state, z_state, B * H, L, d_v, flags,
                              static_cast<cudaStream_t>(cuda_stream));
}

based_status based_prefill(const void* q, const void* k, const void* v, void* out, float* kv_state, float* z_state,
                           int B, int H, int L, int d_feat, int d_v, based_dtype io, int flags, void* workspace,
                           size_t workspace_bytes, void* cuda_stream) {
    return prefill_impl(q, k, v, out, kv_state, z_state, B, H, L, d_feat, d_v, io, flags, workspace, workspace_bytes,
                        cuda_stream, false);
}

based_status based_prefill_f32_parts(const float* q, const float* k, const float* v, float* out, int B, int H, int L, int d_feat,
                                     int d_v, int flags, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!q || !k || !v || !out || B <= 0 || H <= 0 || L <= 0) return BASED_ERR_INVALID_ARG;
    if (flags & ~BASED_NUMERATOR_ONLY) return BASED_ERR_INVALID_ARG;
    if (out == q || out == k || out == v) return BASED_ERR_INVALID_ARG;
    const size_t need = based_f32_parts_bytes(B, H, L, d_feat, d_v, 0);
    if (need == 0 || (long long)B * H > kHeadSlab) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(workspace)) return BASED_ERR_ALIGNMENT;
    if (!workspace || workspace_bytes < need) return BASED_ERR_WORKSPACE;
    return launch_quadratic_forward_f32(q, k, v, out, workspace, B * H, L, d_v, (flags & BASED_NUMERATOR_ONLY) ? 1 : 0,
                                        static_cast<cudaStream_t>(cuda_stream));
}

size_t based_prefill_state_workspace_bytes(int B, int H, int L, int d_feat, int d_v, based_dtype io) {
    if (B <= 0 || H <= 0 || L <= 0 || d_feat != kDFeat || !dv_ok(d_v) || io != BASED_BF16) return 0;
    if ((long long)B * H > kHeadSlab) return prefill_tc_state_workspace_bytes((int)kHeadSlab, L, d_v);   // heads x one partial state: the largest slab's
    return prefill_tc_state_workspace_bytes(B * H, L, d_v);
}

based_status based_prefill_state(const void* k, const void* v, float* kv_state, float* z_state, int B, int H, int L,
                                 int d_feat, int d_v, based_dtype io, int flags, void* workspace,
                                 size_t workspace_bytes, void* cuda_stream) {
    if (!k || !v || !kv_state || !z_state || B <= 0 || H <= 0 || L <= 0) return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (flags & ~(BASED_STATE_CONTINUE | BASED_STATE_SYM)) return BASED_ERR_INVALID_ARG;
    if ((d_feat != kDFeat && !df_generic(d_feat)) || !dv_ok(d_v)) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    const bool tc16 = d_feat == kDFeat && io == BASED_BF16;
    if ((flags & BASED_STATE_SYM) && !tc16) return BASED_ERR_UNSUPPORTED;      // symmetric rows: d' = 16, bf16 io
    if (!aligned16(k) || !aligned16(v) || !aligned16(kv_state) || !aligned16(z_state) || !aligned16(workspace))
        return BASED_ERR_ALIGNMENT;
    if ((long long)B * H > kHeadSlab) {
        const size_t es = esize(io), rows = (flags & BASED_STATE_SYM) ? kDSym : 1 + d_feat + d_feat * d_feat;
        for (long long h0 = 0; h0 < (long long)B * H; h0 += kHeadSlab) {
            const int n = (int)((long long)B * H - h0 < kHeadSlab ? (long long)B * H - h0 : kHeadSlab);
            const based_status st = based_prefill_state(
                off(k, (size_t)h0 * L * d_feat * es), off(v, (size_t)h0 * L * d_v * es), off(kv_state, (size_t)h0 * rows * d_v),
                off(z_state, (size_t)h0 * rows), 1, n, L, d_feat, d_v, io, flags, workspace, workspace_bytes, cuda_stream);
            if (st != BASED_OK) return st;
        }
        return BASED_OK;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (tc16) {
        if (!workspace || workspace_bytes < based_prefill_state_workspace_bytes(B, H, L, d_feat, d_v, io))
            return BASED_ERR_WORKSPACE;
        return launch_prefill_tc_state(k, v, kv_state, z_state, B * H, L, d_v, flags, workspace, stream);
    }
    return launch_state_generic(k, v, kv_state, z_state, B * H, L, d_feat, d_v, io,
                                (flags & BASED_STATE_CONTINUE) ? 1 : 0, stream);
}

based_status based_decode_step(const void* q, const void* k, const void* v, float* kv_state, float* z_state,
                               void* out, int B, int H, int d_feat, int d_v, based_dtype io, void* cuda_stream) {
    if (!q || !k || !v || !out || !kv_state || !z_state || B <= 0 || H <= 0) return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if ((d_feat != kDFeat && !df_generic(d_feat)) || !dv_ok(d_v)) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(kv_state) ||
        !aligned16(z_state))
        return BASED_ERR_ALIGNMENT;
    if (d_feat != kDFeat)
        return launch_decode_generic(q, k, v, kv_state, z_state, out, B * H, d_feat, d_v, io, false,
                                     static_cast<cudaStream_t>(cuda_stream));
    return launch_decode(q, k, v, kv_state, z_state, out, B * H, d_v, io, false, false,
                         static_cast<cudaStream_t>(cuda_stream));
}

based_status based_decode_step_flags(const void* q, const void* k, const void* v, float* kv_state, float* z_state,
                                     void* out, int B, int H, int d_feat, int d_v, based_dtype io, int flags,
                                     void* cuda_stream) {
    if (!q || !k || !v || !out || !kv_state || !z_state || B <= 0 || H <= 0) return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (flags & ~(BASED_STATE_SYM | BASED_NUMERATOR_ONLY)) return BASED_ERR_INVALID_ARG;
    if ((d_feat != kDFeat && !df_generic(d_feat)) || !dv_ok(d_v)) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(kv_state) ||
        !aligned16(z_state))
        return BASED_ERR_ALIGNMENT;
    if (d_feat != kDFeat) {
        if (flags & BASED_STATE_SYM) return BASED_ERR_UNSUPPORTED;
        return launch_decode_generic(q, k, v, kv_state, z_state, out, B * H, d_feat, d_v, io,
                                     (flags & BASED_NUMERATOR_ONLY) != 0, static_cast<cudaStream_t>(cuda_stream));
    }
    return launch_decode(q, k, v, kv_state, z_state, out, B * H, d_v, io, (flags & BASED_STATE_SYM) != 0,
                         (flags & BASED_NUMERATOR_ONLY) != 0, static_cast<cudaStream_t>(cuda_stream));
}

based_status based_decode_step_sym(const void* q, const void* k, const void* v, float* kv_sym, float* z_sym,
                                   void* out, int B, int H, int d_feat, int d_v, based_dtype io,
                                   void* cuda_stream) {
    if (!q || !k || !v || !out || !kv_sym || !z_sym || B <= 0 || H <= 0) return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (d_feat != kDFeat || !dv_ok(d_v)) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(kv_sym) ||
        !aligned16(z_sym))
        return BASED_ERR_ALIGNMENT;
    return launch_decode(q, k, v, kv_sym, z_sym, out, B * H, d_v, io, true, false,
                         static_cast<cudaStream_t>(cuda_stream));
}

static based_status state_convert(const float* kv_in, const float* z_in, float* kv_out, float* z_out, int B, int H,
                                  int d_feat, int d_v, bool to_sym, void* cuda_stream) {
    if (!kv_in || !z_in || !kv_out || !z_out || B <= 0 || H <= 0) return BASED_ERR_INVALID_ARG;
    if (kv_in == kv_out || z_in == z_out) return BASED_ERR_INVALID_ARG;
    if (d_feat != kDFeat || !dv_ok(d_v)) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(kv_in) || !aligned16(z_in) || !aligned16(kv_out) || !aligned16(z_out)) return BASED_ERR_ALIGNMENT;
    return launch_state_convert(kv_in, z_in, kv_out, z_out, B * H, d_v, to_sym,
                                static_cast<cudaStream_t>(cuda_stream));
}

based_status based_state_to_sym(const float* kv_state, const float* z_state, float* kv_sym, float* z_sym, int B,
                                int H, int d_feat, int d_v, void* cuda_stream) {
    return state_convert(kv_state, z_state, kv_sym, z_sym, B, H, d_feat, d_v, true, cuda_stream);
}

based_status based_state_from_sym(const float* kv_sym, const float* z_sym, float* kv_state, float* z_state, int B,
                                  int H, int d_feat, int d_v, void* cuda_stream) {
    return state_convert(kv_sym, z_sym, kv_state, z_state, B, H, d_feat, d_v, false, cuda_stream);
}

based_status swa_forward(const void* q, const void* k, const void* v, void* out, int B, int H, int L, int d,
                         int window, float softmax_scale, based_dtype io, void* cuda_stream) {
    if (!q || !k || !v || !out || B <= 0 || H <= 0 || L <= 0 || window <= 0) return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (out == q || out == k || out == v) return BASED_ERR_INVALID_ARG;
    if (d != 64 || window > 128) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out)) return BASED_ERR_ALIGNMENT;
    if ((long long)B * H > kHeadSlab) {
        const size_t hb = (size_t)L * d * esize(io);
        for (long long h0 = 0; h0 < (long long)B * H; h0 += kHeadSlab) {
            const int n = (int)((long long)B * H - h0 < kHeadSlab ? (long long)B * H - h0 : kHeadSlab);
            const based_status st = swa_forward(off(q, h0 * hb), off(k, h0 * hb), off(v, h0 * hb), off(out, h0 * hb), 1, n, L,
                                                d, window, softmax_scale, io, cuda_stream);
            if (st != BASED_OK) return st;
        }
        return BASED_OK;
    }
    const float scale = softmax_scale > 0.f ? softmax_scale : 0.125f;   // 1/sqrt(64)
    if (io == BASED_BF16 && swa_tc_supported(window))
        return launch_swa_tc(q, k, v, out, B * H, L, window, scale, static_cast<cudaStream_t>(cuda_stream));
    return launch_swa_simt(q, k, v, out, B * H, L, window, scale, io, static_cast<cudaStream_t>(cuda_stream));
}

based_status swa_decode_step(const void* q, const void* k, const void* v, void* k_cache, void* v_cache, void* out,
                             int B, int H, int d, int window, int pos, float softmax_scale, based_dtype io,
                             void* cuda_stream) {
    if (!q || !k || !v || !k_cache || !v_cache || !out || B <= 0 || H <= 0 || window <= 0 || pos < 0)
        return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (d != 64 || window > 128) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(k_cache) || !aligned16(v_cache) ||
        !aligned16(out))
        return BASED_ERR_ALIGNMENT;
    const float scale = softmax_scale > 0.f ? softmax_scale : 0.125f;   // 1/sqrt(64)
    return launch_swa_decode(q, k, v, k_cache, v_cache, out, B * H, window, pos, nullptr, nullptr, scale, io,
                             static_cast<cudaStream_t>(cuda_stream));
}

based_status swa_decode_step_at(const void* q, const void* k, const void* v, void* k_cache, void* v_cache,
                                void* out, int B, int H, int d, int window, const int* pos_device,
                                float softmax_scale, based_dtype io, void* cuda_stream) {
    if (!q || !k || !v || !k_cache || !v_cache || !out || !pos_device || B <= 0 || H <= 0 || window <= 0)
        return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (d != 64 || window > 128) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(k_cache) || !aligned16(v_cache) ||
        !aligned16(out) || (reinterpret_cast<uintptr_t>(pos_device) & 3u))
        return BASED_ERR_ALIGNMENT;
    const float scale = softmax_scale > 0.f ? softmax_scale : 0.125f;   // 1/sqrt(64)
    return launch_swa_decode(q, k, v, k_cache, v_cache, out, B * H, window, 0, pos_device, nullptr, scale, io,
                             static_cast<cudaStream_t>(cuda_stream));
}

based_status swa_decode_step_ragged(const void* q, const void* k, const void* v, void* k_cache, void* v_cache,
                                    void* out, int B, int H, int d, int window, const int* pos_per_sequence,
                                    float softmax_scale, based_dtype io, void* cuda_stream) {
    if (!q || !k || !v || !k_cache || !v_cache || !out || !pos_per_sequence || B <= 0 || H <= 0 || window <= 0)
        return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (d != 64 || window > 128) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(k_cache) || !aligned16(v_cache) ||
        !aligned16(out) || (reinterpret_cast<uintptr_t>(pos_per_sequence) & 3u))
        return BASED_ERR_ALIGNMENT;
    const float scale = softmax_scale > 0.f ? softmax_scale : 0.125f;   // 1/sqrt(64)
    return launch_swa_decode(q, k, v, k_cache, v_cache, out, B * H, window, 0, pos_per_sequence, nullptr, scale, io,
                             static_cast<cudaStream_t>(cuda_stream), H);
}

based_status swa_decode_step_advance(const void* q, const void* k, const void* v, void* k_cache, void* v_cache,
                                     void* out, int B, int H, int d, int window, int* pos_state,
                                     float softmax_scale, based_dtype io, void* cuda_stream) {
    if (!q || !k || !v || !k_cache || !v_cache || !out || !pos_state || B <= 0 || H <= 0 || window <= 0)
        return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (d != 64 || window > 128) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(k_cache) || !aligned16(v_cache) ||
        !aligned16(out) || (reinterpret_cast<uintptr_t>(pos_state) & 7u))
        return BASED_ERR_ALIGNMENT;
    const float scale = softmax_scale > 0.f ? softmax_scale : 0.125f;   // 1/sqrt(64)
    return launch_swa_decode(q, k, v, k_cache, v_cache, out, B * H, window, 0, pos_state, pos_state, scale, io,
                             static_cast<cudaStream_t>(cuda_stream));
}

static based_status generation_step_check(const void* q, const void* k, const void* v, const float* kv_state, const float* z_state,
                                          const void* out, const void* qw, const void* kw, const void* vw, const void* k_cache,
                                          const void* v_cache, const void* out_w, int B, int H, int d_feat, int d_v, int H_w, int d_w,
                                          int window, const int* pos_state, based_dtype io, int flags) {
    if (!q || !k || !v || !kv_state || !z_state || !out || !qw || !kw || !vw || !k_cache || !v_cache || !out_w ||
        !pos_state || B <= 0 || H <= 0 || H_w <= 0 || window <= 0)
        return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (flags & ~(BASED_STATE_SYM | BASED_NUMERATOR_ONLY)) return BASED_ERR_INVALID_ARG;
    if (d_feat != kDFeat || !dv_ok(d_v) || d_w != 64 || window > 128) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H + ((long long)B * H_w + 1) / 2 > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(kv_state) || !aligned16(z_state) ||
        !aligned16(out) || !aligned16(qw) || !aligned16(kw) || !aligned16(vw) || !aligned16(k_cache) ||
        !aligned16(v_cache) || !aligned16(out_w) || (reinterpret_cast<uintptr_t>(pos_state) & 7u))
        return BASED_ERR_ALIGNMENT;
    return BASED_OK;
}

based_status based_generation_step(const void* q, const void* k, const void* v, float* kv_state, float* z_state,
                                   void* out, const void* qw, const void* kw, const void* vw, void* k_cache,
                                   void* v_cache, void* out_w, int B, int H, int d_feat, int d_v, int H_w, int d_w,
                                   int window, int* pos_state, float softmax_scale, based_dtype io, int flags,
                                   void* cuda_stream) {
    const based_status st = generation_step_check(q, k, v, kv_state, z_state, out, qw, kw, vw, k_cache, v_cache, out_w, B, H, d_feat,
                                                  d_v, H_w, d_w, window, pos_state, io, flags);
    if (st != BASED_OK) return st;
    const float scale = softmax_scale > 0.f ? softmax_scale : 0.125f;   // 1/sqrt(64)
    return launch_generation_step(q, k, v, kv_state, z_state, out, B * H, d_v, (flags & BASED_STATE_SYM) != 0,
                                  (flags & BASED_NUMERATOR_ONLY) != 0, qw, kw, vw, k_cache, v_cache, out_w, B * H_w,
                                  window, pos_state, scale, io, static_cast<cudaStream_t>(cuda_stream));
}

// The step's arguments, and the order of its launches.  The kernel is launched as based_generation_step's is, not as a node of
// an instantiated graph: a dependent launch is on the SMs while the one before it drains, which graph launches, each behind
// the end of the one before, are not (16 heads x batch 8 / 16 / 32, 153 rows, d_v 128, on states from memory: 10.5 -> 8.3,
// 13.5 -> 10.2, 20.3 -> 16.8 us per step).  What a graph's launches give besides, an order among themselves whichever streams
// they are on, an event behind every step keeps.
struct based_generation_graph {
    std::vector<unsigned char> args;           // launch_generation_args
    void* buffers[6] = {};
    bool own_inputs = false;                   // the arguments point at inputs other than the buffers
    cudaEvent_t done = nullptr;                // behind the last step
    unsigned long long last_stream = 0;        // its stream's number, which no later stream is given again
    bool launched = false;
    std::mutex mu;
};

void based_generation_graph_destroy(based_generation_graph* g) {
    if (!g) return;
    if (g->done) cudaEventDestroy(g->done);
    delete g;
}

based_status based_generation_graph_create(void* q, void* k, void* v, float* kv_state, float* z_state, void* out, void* qw,
                                           void* kw, void* vw, void* k_cache, void* v_cache, void* out_w, int B, int H,
                                           int d_feat, int d_v, int H_w, int d_w, int window, int* pos_state,
                                           float softmax_scale, based_dtype io, int flags, based_generation_graph** graph) {
    if (!graph) return BASED_ERR_INVALID_ARG;
    *graph = nullptr;
    const based_status st = generation_step_check(q, k, v, kv_state, z_state, out, qw, kw, vw, k_cache, v_cache, out_w, B, H, d_feat,
                                                  d_v, H_w, d_w, window, pos_state, io, flags);
    if (st != BASED_OK) return st;
    based_generation_graph* g = new (std::nothrow) based_generation_graph;
    if (!g) return BASED_ERR_CUDA;
    const float scale = softmax_scale > 0.f ? softmax_scale : 0.125f;   // 1/sqrt(64)
    try {
        g->args.resize(generation_step_args_bytes());
    } catch (const std::bad_alloc&) {
        delete g;
        return BASED_ERR_CUDA;
    }
    if (make_generation_args(g->args.data(), q, k, v, kv_state, z_state, out, B * H, d_v, (flags & BASED_STATE_SYM) != 0,
                             (flags & BASED_NUMERATOR_ONLY) != 0, qw, kw, vw, k_cache, v_cache, out_w, B * H_w, window, pos_state,
                             scale, io) != BASED_OK ||
        cudaEventCreateWithFlags(&g->done, cudaEventDisableTiming) != cudaSuccess) {
        based_generation_graph_destroy(g);
        return BASED_ERR_CUDA;
    }
    void* const buffers[6] = {q, k, v, qw, kw, vw};
    for (int i = 0; i < 6; ++i) g->buffers[i] = buffers[i];
    *graph = g;
    return BASED_OK;
}

based_status based_generation_graph_step(based_generation_graph* g, const void* q, const void* k, const void* v, const void* qw,
                                         const void* kw, const void* vw, void* cuda_stream) {
    if (!g) return BASED_ERR_INVALID_ARG;
    const void* const in[6] = {q, k, v, qw, kw, vw};
    int given = 0;
    for (const void* p : in) {
        given += p != nullptr;
        if (!aligned16(p)) return BASED_ERR_ALIGNMENT;
    }
    if (given != 0 && given != 6) return BASED_ERR_INVALID_ARG;
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    // a stream under capture cannot take the order among the steps (nor could it take a graph launch)
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    if (cudaStreamIsCapturing(stream, &capture) != cudaSuccess || capture != cudaStreamCaptureStatusNone ||
        cudaStreamGetId(stream, &id) != cudaSuccess)
        return BASED_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g->mu);
    if (given || g->own_inputs) {
        generation_step_inputs(g->args.data(), in, g->buffers);
        g->own_inputs = given != 0;
    }
    if (g->launched && id != g->last_stream && cudaStreamWaitEvent(stream, g->done, 0) != cudaSuccess) return BASED_ERR_CUDA;
    const based_status st = launch_generation_args(g->args.data(), stream);
    if (st != BASED_OK) return st;
    g->launched = true;
    g->last_stream = id;
    return cudaEventRecord(g->done, stream) == cudaSuccess ? BASED_OK : BASED_ERR_CUDA;
}

static based_status baseconv_check(const void* a, const void* g, const float* h, const float* b2, const void* out,
                                   int B, int N, int C, int width, based_dtype io) {
    if (!a || !g || !h || !b2 || !out || B <= 0 || N <= 0 || C <= 0 || width <= 0) return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (out == g) return BASED_ERR_INVALID_ARG;
    if (width > 4 || C % 8 != 0 || B > 65535 || (N + 63) / 64 > 65535) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(a) || !aligned16(g) || !aligned16(h) || !aligned16(b2) || !aligned16(out)) return BASED_ERR_ALIGNMENT;
    return BASED_OK;
}

based_status baseconv_gate_forward(const void* a, const void* g, const float* h, const float* b2, void* out, int B,
                                   int N, int C, int width, based_dtype io, void* cuda_stream) {
    const based_status st = baseconv_check(a, g, h, b2, out, B, N, C, width, io);
    if (st != BASED_OK) return st;
    return launch_baseconv(a, g, h, b2, nullptr, out, B, N, C, width, false, io,
                           static_cast<cudaStream_t>(cuda_stream));
}

based_status baseconv_gate_step(const void* a, const void* g, const float* h, const float* b2, void* conv_state,
                                void* out, int B, int C, int width, based_dtype io, void* cuda_stream) {
    const based_status st = baseconv_check(a, g, h, b2, out, B, 1, C, width, io);
    if (st != BASED_OK) return st;
    if (width > 1 && !conv_state) return BASED_ERR_INVALID_ARG;
    if (!aligned16(conv_state)) return BASED_ERR_ALIGNMENT;
    return launch_baseconv(a, g, h, b2, conv_state, out, B, 1, C, width, true, io,
                           static_cast<cudaStream_t>(cuda_stream));
}

size_t based_prefill_backward_workspace_bytes(int B, int H, int L, int d_v, based_dtype io) {
    if (B <= 0 || H <= 0 || L <= 0 || !dv_ok(d_v)) return 0;
    const int heads = (long long)B * H > kHeadSlab ? (int)kHeadSlab : B * H;       // the largest slab of heads
    if (io == BASED_BF16) return backward_tc_workspace_bytes(heads, L, d_v);
    return (size_t)heads * L * 2 * sizeof(float);
}

int based_prefill_backward_block_tokens(int B, int H, int L, int d_feat, int d_v, based_dtype io, int flags,
                                        int with_out) {
    if (B <= 0 || H <= 0 || L <= 0 || !dv_ok(d_v) || io != BASED_BF16) return 0;
    return backward_tc_block_tokens(B * H, L, d_feat, d_v, (with_out || (flags & BASED_NUMERATOR_ONLY)) ? 1 : 0);
}

// fp32 io, one slab of heads, checked arguments; dout_H: 0, or H where dout lies [B, L, H, d_v]
static based_status backward_f32(const void* q, const void* k, const void* v, const void* dout, int dout_H, void* dq, void* dk,
                                 void* dv, int B, int H, int L, int d_v, int flags, void* workspace, size_t workspace_bytes,
                                 void* cuda_stream) {
    auto in = [](const void* p) { return static_cast<const float*>(p); };
    auto out = [](void* p) { return static_cast<float*>(p); };
    const int numerator_only = (flags & BASED_NUMERATOR_ONLY) ? 1 : 0;
    const size_t parts = based_f32_parts_bytes(B, H, L, kDFeat, d_v, 1);
    if (parts > 0 && workspace_bytes >= parts)
        return launch_quadratic_backward_f32(in(q), in(k), in(v), in(dout), dout_H, out(dq), out(dk), out(dv), workspace, B * H, L,
                                             numerator_only, static_cast<cudaStream_t>(cuda_stream));
    return launch_prefill_backward_f32(in(q), in(k), in(v), in(dout), dout_H, out(dq), out(dk), out(dv), out(workspace), B * H, L,
                                       d_v, numerator_only, static_cast<cudaStream_t>(cuda_stream));
}

static based_status prefill_backward(const void* q, const void* k, const void* v, const void* out, const void* dout,
                                     void* dq, void* dk, void* dv, int B, int H, int L, int d_feat, int d_v,
                                     based_dtype io, int flags, void* workspace, size_t workspace_bytes,
                                     void* cuda_stream) {
    if (!q || !k || !v || !dout || !dq || !dk || !dv || B <= 0 || H <= 0 || L <= 0) return BASED_ERR_INVALID_ARG;
    if (io != BASED_F32 && io != BASED_BF16) return BASED_ERR_INVALID_ARG;
    if (flags & ~BASED_NUMERATOR_ONLY) return BASED_ERR_INVALID_ARG;
    if (dq == q || dq == k || dk == q || dk == k || dv == v || dv == dout) return BASED_ERR_INVALID_ARG;
    // the other feature dimensions: bf16 io only (the tensor-core kernels take d' as a parameter)
    if (!(d_feat == kDFeat || (df_generic(d_feat) && io == BASED_BF16)) || !dv_ok(d_v)) return BASED_ERR_UNSUPPORTED;
    if ((long long)B * H > 0x7fffffffLL) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(dout) || !aligned16(dq) || !aligned16(dk) ||
        !aligned16(dv) || !aligned16(workspace) || !aligned16(out))
        return BASED_ERR_ALIGNMENT;
    if (!workspace || workspace_bytes < based_prefill_backward_workspace_bytes(B, H, L, d_v, io))
        return BASED_ERR_WORKSPACE;
    if ((long long)B * H > kHeadSlab) {
        const size_t qb = (size_t)L * d_feat * esize(io), vb = (size_t)L * d_v * esize(io);
        for (long long h0 = 0; h0 < (long long)B * H; h0 += kHeadSlab) {
            const int n = (int)((long long)B * H - h0 < kHeadSlab ? (long long)B * H - h0 : kHeadSlab);
            const based_status st = prefill_backward(off(q, h0 * qb), off(k, h0 * qb), off(v, h0 * vb), off(out, h0 * vb),
                                                     off(dout, h0 * vb), off(dq, h0 * qb), off(dk, h0 * qb), off(dv, h0 * vb), 1,
                                                     n, L, d_feat, d_v, io, flags, workspace, workspace_bytes, cuda_stream);
            if (st != BASED_OK) return st;
        }
        return BASED_OK;
    }
    if (io == BASED_BF16)
        return launch_prefill_backward_tc(q, k, v, out, dout, 0, dq, dk, dv, static_cast<float*>(workspace), B * H, L,
                                          d_feat, d_v, (flags & BASED_NUMERATOR_ONLY) ? 1 : 0,
                                          static_cast<cudaStream_t>(cuda_stream));
    return backward_f32(q, k, v, dout, 0, dq, dk, dv, B, H, L, d_v, flags, workspace, workspace_bytes, cuda_stream);
}

based_status based_prefill_backward(const void* q, const void* k, const void* v, const void* dout, void* dq,
                                    void* dk, void* dv, int B, int H, int L, int d_feat, int d_v, based_dtype io,
                                    int flags, void* workspace, size_t workspace_bytes, void* cuda_stream) {
    return prefill_backward(q, k, v, nullptr, dout, dq, dk, dv, B, H, L, d_feat, d_v, io, flags, workspace,
                            workspace_bytes, cuda_stream);
}

based_status based_prefill_backward_with_out(const void* q, const void* k, const void* v, const void* out,
                                             const void* dout, void* dq, void* dk, void* dv, int B, int H, int L,
                                             int d_feat, int d_v, based_dtype io, int flags, void* workspace,
                                             size_t workspace_bytes, void* cuda_stream) {
    if (!out || out == dq || out == dk || out == dv) return BASED_ERR_INVALID_ARG;
    return prefill_backward(q, k, v, out, dout, dq, dk, dv, B, H, L, d_feat, d_v, io, flags, workspace,
                            workspace_bytes, cuda_stream);
}

based_status based_prefill_backward_tokens_first(const void* q, const void* k, const void* v, const void* dout, void* dq, void* dk,
                                                 void* dv, int B, int H, int L, int d_feat, int d_v, based_dtype io, int flags,
                                                 void* workspace, size_t workspace_bytes, void* cuda_stream) {
    if (!q || !k || !v || !dout || !dq || !dk || !dv || B <= 0 || H <= 0 || L <= 0) return BASED_ERR_INVALID_ARG;
    if (flags & ~BASED_NUMERATOR_ONLY) return BASED_ERR_INVALID_ARG;
    if (dq == q || dq == k || dk == q || dk == k || dv == v || dv == dout) return BASED_ERR_INVALID_ARG;
    // one slab of heads, rows counted in 32 bits
    if (io != BASED_F32 || d_feat != kDFeat || !dv_ok(d_v) || (long long)B * H > kHeadSlab || (long long)B * H * L > 0x7fffffffLL)
        return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(dout) || !aligned16(dq) || !aligned16(dk) || !aligned16(dv) ||
        !aligned16(workspace))
        return BASED_ERR_ALIGNMENT;
    if (!workspace || workspace_bytes < based_prefill_backward_workspace_bytes(B, H, L, d_v, io)) return BASED_ERR_WORKSPACE;
    return backward_f32(q, k, v, dout, H, dq, dk, dv, B, H, L, d_v, flags, workspace, workspace_bytes, cuda_stream);
}

based_status based_prefill_backward_tokens_first_with_out(const void* q, const void* k, const void* v, const void* out,
                                                          const void* dout, void* dq, void* dk, void* dv, int B, int H, int L,
                                                          int d_feat, int d_v, based_dtype io, int flags, void* workspace,
                                                          size_t workspace_bytes, void* cuda_stream) {
    if (!q || !k || !v || !out || !dout || !dq || !dk || !dv || B <= 0 || H <= 0 || L <= 0) return BASED_ERR_INVALID_ARG;
    if (flags & ~BASED_NUMERATOR_ONLY) return BASED_ERR_INVALID_ARG;
    if (dq == q || dq == k || dk == q || dk == k || dv == v || dv == dout || out == dq || out == dk || out == dv) return BASED_ERR_INVALID_ARG;
    // one slab of heads, rows counted in 32 bits
    if (io != BASED_BF16 || !(d_feat == kDFeat || df_generic(d_feat)) || !dv_ok(d_v) || (long long)B * H > kHeadSlab ||
        (long long)B * H * L > 0x7fffffffLL)
        return BASED_ERR_UNSUPPORTED;
    if (!aligned16(q) || !aligned16(k) || !aligned16(v) || !aligned16(out) || !aligned16(dout) || !aligned16(dq) || !aligned16(dk) ||
        !aligned16(dv) || !aligned16(workspace))
        return BASED_ERR_ALIGNMENT;
    if (!workspace || workspace_bytes < based_prefill_backward_workspace_bytes(B, H, L, d_v, io)) return BASED_ERR_WORKSPACE;
    return launch_prefill_backward_tc(q, k, v, out, dout, H, dq, dk, dv, static_cast<float*>(workspace), B * H, L, d_feat, d_v,
                                      (flags & BASED_NUMERATOR_ONLY) ? 1 : 0, static_cast<cudaStream_t>(cuda_stream));
}

based_status based_tokens_to_heads(const void* src, void* dst, int B, int H, int L, int row_bytes, void* cuda_stream) {
    if (!src || !dst || src == dst || B <= 0 || H <= 0 || L <= 0 || row_bytes <= 0) return BASED_ERR_INVALID_ARG;
    // one head of one sequence is indexed with 32 bits, heads and sequences by the grid's y and z
    if (row_bytes % 16 || (long long)L * (row_bytes / 16) > 0x7fffffffLL || B > 65535 || H > 65535) return BASED_ERR_UNSUPPORTED;
    if (!aligned16(src) || !aligned16(dst)) return BASED_ERR_ALIGNMENT;
    return launch_tokens_to_heads(src, dst, B, H, L, row_bytes, static_cast<cudaStream_t>(cuda_stream));
}

based_status based_preload_decode(void) {
    unsigned int* err = nullptr;
    based_status st = error_word_ptr(&err);
    if (st == BASED_OK) st = preload_decode();
    if (st == BASED_OK) st = preload_swa_decode();
    if (st == BASED_OK) st = preload_generation_step();
    return st;
}

based_status based_poll_error(void* cuda_stream) {
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(cuda_stream)) != cudaSuccess) return BASED_ERR_CUDA;
    unsigned int word = 0;
    if (cudaMemcpyFromSymbol(&word, g_error_word, sizeof(word)) != cudaSuccess) return BASED_ERR_CUDA;
    if (word != 0) {
        const unsigned int zero = 0;
        if (cudaMemcpyToSymbol(g_error_word, &zero, sizeof(zero)) != cudaSuccess) return BASED_ERR_CUDA;
        return BASED_ERR_DEVICE_TIMEOUT;
    }
    return BASED_OK;
}

}  // extern "C"

namespace based {
based_status prefill_fit_workspace(const void* q, const void* k, const void* v, void* out, float* kv_state, float* z_state,
                                   int B, int H, int L, int d_feat, int d_v, based_dtype io, int flags, void* workspace,
                                   size_t workspace_bytes, void* cuda_stream) {
    return ::prefill_impl(q, k, v, out, kv_state, z_state, B, H, L, d_feat, d_v, io, flags, workspace, workspace_bytes,
                          cuda_stream, true);
}
}  // namespace based
