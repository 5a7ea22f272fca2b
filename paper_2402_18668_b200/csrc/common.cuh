// Shared host/device helpers of libbased (sm_100a only).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>

#include "based.h"

namespace based {

constexpr int kDFeat = 16;                              // d' of the paper
constexpr int kD = 1 + kDFeat + kDFeat * kDFeat;        // 273 expanded features
constexpr int kDSym = 1 + kDFeat + kDFeat * (kDFeat + 1) / 2;   // 153 features, one per unordered pair
constexpr int kSMs = 148;                                // B200
constexpr float kEps = 1e-12f;                          // eps of the paper's listings
// feature-map scales: x / d'^(1/4) and x_m x_n / (sqrt(2) sqrt(d')), d' = 16
constexpr float kLinScale = 0.5f;
constexpr float kQuadScale = 0.17677669529663687f;      // 1 / (4 sqrt 2)

// Device address of the sticky status word of the current device (bit 0: a bounded
// wait timed out).  Kernels that can time out receive it as an argument.
based_status error_word_ptr(unsigned int** ptr);

// serialises the per-device one-time set-up of the launchers (function attributes and the like)
std::mutex& setup_mutex();

// host-side bookkeeping
void note_launch();                                     // ++launch counter
based_status check_launch(const char* what);            // cudaGetLastError -> status

// Launch, PARTS > 1 CTAs per cluster; dependent: with programmatic stream serialization, so that the grid's CTAs may be
// scheduled once every CTA of the grid ahead in the stream has signalled (griddepcontrol.launch_dependents) or left.  The
// kernel itself waits (enter_dependent) before it touches what that grid reads or writes; behind a kernel that never signals
// such a launch behaves like a plain one.
template <typename... P, typename... A>
cudaError_t launch_ex(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, int cluster, bool dependent, cudaStream_t stream,
                      const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at[2]{};
    int n = 0;
    if (dependent) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        at[n].id = cudaLaunchAttributeClusterDimension;
        at[n].val.clusterDim.x = cluster;
        at[n].val.clusterDim.y = 1;
        at[n++].val.clusterDim.z = 1;
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
// Whether the definition form's forward, `tiles` CTAs of up to n = `per_head` turns of its loop each on the chip's `slots`, is a dependent
// launch.  One that nearly fills the slots once is not: its first CTAs, the longest, would double up on the SMs that the grid ahead
// leaves first (us repeated, dependent / plain.  d' 8 d_v 64, two CTAs per SM: 16 heads L2048 16.3 / 14.1, 20 L1409 12.6 / 11.2, 10 L4096 29 /
// 24; four: 64 L777 14.3 / 12.5, 64 L1100 19.6 / 16.4, 20 L4096 55 / 45; d_v 128: 16 L2048 19.9 / 18.4, 10 L4096 35.6 / 31.6).  Otherwise the
// set-up beside that grid pays: few tiles (16 L1024 7.5 / 8.1), short loops (128 L200 5.3 / 6.1, 100 L777 15.8 / 17.0), more than a wave (the
// longer the loops the later: 32 L2048 19.8 / 21.5, 64 L2048 34 / 36, 28 L4096 53.5 / 52.6).
inline bool dependent_forward(long long tiles, int per_head, int slots) {
    return per_head < 7 || 3 * tiles <= 2 * slots || 64 * (tiles - slots) > (long long)(per_head - 4) * slots;
}
// Splits an SM's 256 KB between L1 and shared memory for a kernel that streams through L1: loads in flight take L1 lines, and
// without a preference a kernel runs with whatever split the one before it left (decode step, 2048 heads, d_v 128: 91 us
// with a quarter for shared memory or no preference alone, 113 with all of it).  Once per kernel and device.
template <typename K>
cudaError_t prefer_l1(K kernel, int shared_percent, std::atomic<bool> (&done)[64]) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= 64) return e != cudaSuccess ? e : cudaErrorInvalidDevice;
    if (done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    const cudaError_t f = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, shared_percent);
    if (f == cudaSuccess) done[dev].store(true, std::memory_order_release);
    return f;
}
__device__ __forceinline__ void enter_dependent() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename T> __device__ __forceinline__ float to_f32(T x);
template <> __device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// value of expanded feature f (0..272) of a raw 16-vector x held in registers/shared memory
__device__ __forceinline__ float phi_at(const float* x, int f) {
    if (f == 0) return 1.0f;
    if (f <= kDFeat) return x[f - 1] * kLinScale;
    const int p = f - 1 - kDFeat;
    return x[p >> 4] * x[p & 15] * kQuadScale;
}

// Symmetric feature set: index 0 the constant, 1..16 the linear terms, then the pairs m <= n in
// row-major order of the upper triangle.  pair_of(p) returns (m, n) of pair p in [0, 136).
__device__ __forceinline__ void pair_of(int p, int& m, int& n) {
    // m = the largest with 16 m - m (m - 1) / 2 <= p, the root of a quadratic: its argument is a perfect square (and the
    // square root exact) where p starts a row, and at least 8 below the next one elsewhere
    m = static_cast<int>((33.f - sqrtf(1089.f - 8.f * static_cast<float>(p))) * 0.5f);
    n = p - kDFeat * m + m * (m - 1) / 2 + m;
}
// row of pair (m, n), m <= n, in the symmetric layout
__host__ __device__ constexpr int sym_pair_row(int m, int n) {
    return 1 + kDFeat + m * kDFeat - m * (m - 1) / 2 + (n - m);
}
// value of symmetric feature f (0..152): x_m^2 / (4 sqrt 2) on the diagonal, x_m x_n / 4 off it
__device__ __forceinline__ float psi_at(const float* x, int f) {
    if (f == 0) return 1.0f;
    if (f <= kDFeat) return x[f - 1] * kLinScale;
    int m, n;
    pair_of(f - 1 - kDFeat, m, n);
    return x[m] * x[n] * (m == n ? kQuadScale : 0.25f);
}

// kernel launchers (defined in the .cu files; all asynchronous on `stream`)
// sym: the state has the 153 symmetric rows instead of the 273 full ones
based_status launch_decode(const void* q, const void* k, const void* v, float* kv, float* z, void* out,
                           int BH, int d_v, based_dtype io, bool sym, bool numerator_only, cudaStream_t stream);
// both mixers' decode steps of one token in one launch (generation_step.cu)
based_status launch_generation_step(const void* q, const void* k, const void* v, float* kv, float* z, void* out,
                                    int n_lin, int d_v, bool sym, bool numerator_only, const void* qw, const void* kw,
                                    const void* vw, void* kc, void* vc, void* outw, int n_swa, int window,
                                    int* pos_state, float scale, based_dtype io, cudaStream_t stream);
based_status preload_generation_step();
// the same call kept as its arguments (generation_step_args_bytes of them) and launched again and again, each launch no call of
// based_generation_step and not counted as one;
// generation_step_inputs points them at other inputs (null: at `buffers`, q k v qw kw vw) that the step also copies into the buffers
size_t generation_step_args_bytes();
based_status make_generation_args(void* args, const void* q, const void* k, const void* v, float* kv, float* z, void* out,
                                  int n_lin, int d_v, bool sym, bool numerator_only, const void* qw, const void* kw, const void* vw,
                                  void* kc, void* vc, void* outw, int n_swa, int window, int* pos_state, float scale,
                                  based_dtype io);
based_status launch_generation_args(const void* args, cudaStream_t stream);
void generation_step_inputs(void* args, const void* const* inputs, void* const* buffers);
// full (273-row) state -> symmetric (153-row) state, or back
based_status launch_state_convert(const float* kv_in, const float* z_in, float* kv_out, float* z_out, int BH,
                                  int d_v, bool to_sym, cudaStream_t stream);
// fp32 io (prefill_f32.cu)
based_status launch_prefill_f32(const void* q, const void* k, const void* v, void* out, float* kv, float* z, int BH,
                                int L, int d_v, int flags, cudaStream_t stream);
// bf16 tensor-core prefill (tcgen05); workspace holds partial states of sequence segments.  prefill_tc_workspace_bytes
// is what the fastest plan needs; workspace_limit = the bytes behind `workspace`: a call given less takes the fastest
// plan that fits (fewer segments per head, in the end none: the plain loop and the recompute mode need no workspace).
size_t prefill_tc_workspace_bytes(int BH, int L, int d_v);
based_status launch_prefill_tc(const void* q, const void* k, const void* v, void* out, float* kv, float* z, int BH,
                               int L, int d_v, int flags, void* workspace, cudaStream_t stream,
                               size_t workspace_limit = ~(size_t)0);
// based_prefill without its workspace check: the plan is fitted to the workspace given (for based_prefill_static_scratch)
based_status prefill_fit_workspace(const void* q, const void* k, const void* v, void* out, float* kv_state, float* z_state,
                                   int B, int H, int L, int d_feat, int d_v, based_dtype io, int flags, void* workspace,
                                   size_t workspace_bytes, void* cuda_stream);
// bf16 tensor-core sliding window (window <= 128)
bool swa_tc_supported(int window);
based_status launch_swa_tc(const void* q, const void* k, const void* v, void* out, int BH, int L, int window,
                           float scale, cudaStream_t stream);
// pos_dev != nullptr: the position is read from device memory by the kernel (pos is ignored);
// pos_adv != nullptr ({position, ticket}, pos_dev == pos_adv): the kernel also stores position + 1 at its end
based_status launch_swa_decode(const void* q, const void* k, const void* v, void* kc, void* vc, void* out, int BH,
                               int window, int pos, const int* pos_dev, int* pos_adv, float scale, based_dtype io,
                               cudaStream_t stream, int pos_group = 0);
// [B, L, H, row] -> [B, H, L, row]
based_status launch_tokens_to_heads(const void* src, void* dst, int B, int H, int L, int row_bytes, cudaStream_t stream);
// gated short convolution (BaseConv core); step: one token on a [B, width-1, C] state, N ignored
based_status launch_baseconv(const void* a, const void* g, const float* h, const float* b2, void* state, void* out,
                             int B, int N, int C, int width, bool step, based_dtype io, cudaStream_t stream);
// backward of the linear attention (fp32 FMA, quadratic form); stats: [BH, L] float2 scratch
// dout_H: 0, or H where g lies [B, L, H, d_v]
based_status launch_prefill_backward_f32(const float* q, const float* k, const float* v, const float* g, int dout_H, float* dq,
                                         float* dk, float* dv, float* stats, int BH, int L, int d_v, int numerator_only,
                                         cudaStream_t stream);
// fp32 io in definition form on the tensor cores, operands in three bf16 parts (quadratic_f32_tc.cu): outputs from the empty
// state, and the backward pass.  quadratic_f32_workspace_bytes: 0 where the other fp32 kernels are the faster
size_t quadratic_f32_workspace_bytes(int BH, int L, int d_v, bool backward);
based_status launch_quadratic_forward_f32(const float* q, const float* k, const float* v, float* out, void* ws, int BH, int L,
                                          int d_v, int numerator_only, cudaStream_t stream);
// dout_H: 0, or H where g lies [B, L, H, d_v]
based_status launch_quadratic_backward_f32(const float* q, const float* k, const float* v, const float* g, int dout_H, float* dq,
                                           float* dk, float* dv, void* ws, int BH, int L, int numerator_only, cudaStream_t stream);
// feature dimensions 8, 24, 32 (fp32 FMA, definition form); state layout [1 + d' + d'^2, d_v]
based_status launch_prefill_generic(const void* q, const void* k, const void* v, void* out, float* kv, float* z,
                                    int BH, int L, int d_feat, int d_v, based_dtype io, int flags,
                                    cudaStream_t stream);
// the final state of those feature dimensions on tensor cores (bf16 io); cont: add to the state given
based_status launch_state_generic_tc(const void* k, const void* v, float* kv, float* z, int BH, int L, int d_feat,
                                     int d_v, int cont, cudaStream_t stream);
// block_state_tc.cu: block states of the block-wise backward pass (d' = 16, bf16), transposed: st [BH x nblk][d_v][160]
// bf16 and sv [BH x nblk][160]: for every block of W tokens the sums over the blocks before it (rev = 0) or after it
// (rev = 1), one CTA per head; stats: (1 / D, b) per
// token for the query side (x = q, val = dout), null for the key side (x = k, val = v); part, zpart: null, or the
// blocks' own sums in fp32 instead (one CTA per head and block), for state_scan_kernel; val_H: 0, or H where val lies
// [B, L, H, d_v]
based_status launch_block_states_tc(const void* x, const void* val, const void* stats, void* st, float* sv, float* part,
                                    float* zpart, int BH, int val_H, int L, int W, int d_v, int rev, cudaStream_t stream);
// the state of a token block alone (no outputs): kv (+)= sum_j phi(k_j) v_j^T, z (+)= sum_j phi(k_j)
based_status launch_state_generic(const void* k, const void* v, float* kv, float* z, int BH, int L, int d_feat, int d_v,
                                  based_dtype io, int cont, cudaStream_t stream);
size_t prefill_tc_state_workspace_bytes(int BH, int L, int d_v);
based_status launch_prefill_tc_state(const void* k, const void* v, float* kv, float* z, int BH, int L, int d_v,
                                     int flags, void* workspace, cudaStream_t stream);
based_status launch_decode_generic(const void* q, const void* k, const void* v, float* kv, float* z, void* out,
                                   int BH, int d_feat, int d_v, based_dtype io, bool numerator_only,
                                   cudaStream_t stream);
// the same on tensor cores (bf16 io); ws: backward_tc_workspace_bytes
size_t backward_tc_workspace_bytes(int BH, int L, int d_v);
// block length of the block-wise path for this shape, 0 where the tile path runs (merged: forward output given, or
// the numerator-only form)
int backward_tc_block_tokens(int BH, int L, int d_feat, int d_v, int merged);
// out: the forward output (may be null): with it, statistics and dq run as one sweep
// dout_H: 0, or H where g lies [B, L, H, d_v]
based_status launch_prefill_backward_tc(const void* q, const void* k, const void* v, const void* out, const void* g, int dout_H,
                                        void* dq, void* dk, void* dv, float* ws, int BH, int L, int d_feat, int d_v,
                                        int numerator_only, cudaStream_t stream);
// definition-form forward on tensor cores for d' in {8, 24, 32} (bf16 io, empty initial state); overlapped: beside the
// kernel before it in the stream (launch_state_generic_tc's, which lets it), whose results it does not use
based_status launch_quadratic_forward_tc(const void* q, const void* k, const void* v, void* out, int BH, int L,
                                         int d_feat, int d_v, int numerator_only, bool overlapped, cudaStream_t stream);
// the same with two groups of row warps per CTA (quadratic_fwd_tc.cu)
based_status launch_quadratic_groups_tc(const void* q, const void* k, const void* v, void* out, int BH, int L,
                                        int d_feat, int d_v, int numerator_only, bool overlapped, cudaStream_t stream);
// load the generation-step kernels into the current context
based_status preload_decode();
based_status preload_swa_decode();
based_status launch_swa_simt(const void* q, const void* k, const void* v, void* out, int BH, int L, int window,
                             float scale, based_dtype io, cudaStream_t stream);

}  // namespace based
